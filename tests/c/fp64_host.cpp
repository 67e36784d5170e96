// Host build of the two-operation FP64 reciprocal and square root
// (csrc/fp64.cuh) for the CPU tests: the CUDA intrinsics get host definitions,
// the two hardware approximations an exact value off by argv[1] FP32 units
// (the device's are within two).  Prints, per function, the number of cases
// whose error exceeds half a unit of the result by more than 2^-20 of one.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>

template <class To, class From>
static To bits(From x) {
  To y;
  std::memcpy(&y, &x, sizeof y);
  return y;
}
static int g_off = 0;
static float __uint_as_float(unsigned u) { return bits<float>(u); }
static unsigned __float_as_uint(float f) { return bits<unsigned>(f); }
static float __fadd_rn(float a, float b) { return a + b; }
static float __fsub_rn(float a, float b) { return a - b; }
static float __fmul_rn(float a, float b) { return a * b; }
static float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
static float __fdividef(float a, float b) { return __uint_as_float(__float_as_uint(a / b) + g_off); }
static float rsqrtf(float a) { return __uint_as_float(__float_as_uint((float)(1.0 / std::sqrt((double)a))) + g_off); }
static float __uint2float_rn(unsigned u) { return (float)u; }
static unsigned __float2uint_rn(float f) { return (unsigned)std::nearbyintf(f); }
static long long __double_as_longlong(double d) { return bits<long long>(d); }
static double __longlong_as_double(long long l) { return bits<double>(l); }
static int __double2hiint(double d) { return (int)(bits<uint64_t>(d) >> 32); }
static int __double2loint(double d) { return (int)bits<uint64_t>(d); }
static double __hiloint2double(int hi, int lo) { return bits<double>((uint64_t)(unsigned)hi << 32 | (unsigned)lo); }
static unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) { return hi << s | lo >> (32 - s); }
using std::fma;
using std::fmaxf;
using std::sqrt;

#include "fp64.cuh"

static uint64_t g_state = 0x9e3779b97f4a7c15ull;
static uint64_t next_u64() {  // xorshift64*
  g_state ^= g_state >> 12;
  g_state ^= g_state << 25;
  g_state ^= g_state >> 27;
  return g_state * 0x2545f4914f6cdd1dull;
}

static long bad_rcp = 0, bad_sqrt = 0;
static void check(double x) {
  // scaled so that the residuals neither overflow nor lose bits: x = m 2^e
  int e;
  const double m = std::frexp(std::fabs(x), &e), z = std::ldexp(std::fabs(icon::rcp(x)), e);
  const double half = 0.5 * (std::nextafter(z, 4.0) - z) * (1.0 + 0x1p-20);
  if (!(std::fabs(fma(-m, z, 1.0)) <= m * half) || std::signbit(icon::rcp(x)) != std::signbit(x)) ++bad_rcp;
  const double a = std::fabs(x);
  const int h = (e & 1) ? (e + 1) / 2 : e / 2;
  const double q = std::ldexp(a, -2 * h), s = std::ldexp(icon::sqrt2(a), -h);
  const double u = 0.5 * (std::nextafter(s, 4.0) - s) * (1.0 + 0x1p-20);
  if (!(std::fabs(fma(-s, s, q)) <= 2.0 * s * u + u * u)) ++bad_sqrt;
}

int main(int argc, char** argv) {
  g_off = argc > 1 ? std::atoi(argv[1]) : 0;
  for (int i = 0; i < 400000; ++i) {
    const uint64_t r = next_u64();
    const uint64_t ex = 1 + (r >> 52) % 2043;  // below 2^1022
    check(bits<double>((r & 0x800fffffffffffffull) | ex << 52));
    const uint64_t base = bits<uint64_t>(std::ldexp(1.0, (int)(i % 7) - 3));
    check(bits<double>(base + (uint64_t)(i % 4001) - 2000));  // around powers of two
    check(bits<double>(base + (r >> 34)));
  }
  const double inf = INFINITY;
  check(0x1p-1022);
  check(0x1.fffffffffffffp1021);
  const double no_rcp[] = {0.0, -0.0, 0x1p-1040, inf, -inf, NAN, 0x1p1022, 0x1p1023};
  for (double x : no_rcp)
    if (!std::isnan(icon::rcp(x))) ++bad_rcp;
  const double spec[] = {0.0, -0.0, 0x1p-1074, 0x1p-1023, inf, -inf, -1.0, NAN};
  for (double x : spec) {
    const double a = icon::sqrt2(x), b = std::sqrt(x);
    if (std::isnan(b) ? !std::isnan(a) : a != b || std::signbit(a) != std::signbit(b)) ++bad_sqrt;
  }
  std::printf("%ld %ld\n", bad_rcp, bad_sqrt);
  return 0;
}
