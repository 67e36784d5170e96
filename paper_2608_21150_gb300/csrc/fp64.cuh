// FP64 reciprocal and square root in two FP64 operations each.  An FP64
// instruction holds its scheduler for 64 cycles on this GPU, as long as some
// thirty integer or FP32 ones, and bounds the kernels that use them: 1/x took
// three from a double-word seed widened by an addition, a division eight, the
// library's square root about eight.  The argument is scaled by its exponent
// field to [1, 2) (square root: [1, 4)); an FP32 approximation, taken low by a
// few units so that what is missing is positive, is refined in FP32 (Newton)
// to about 2^-42 and joined with its correction as integers; one FP64 residual
// and one multiply-add then give the result within half a unit (and 2^-20 of
// one).  The correction words hold weights of 2^-48 and 2^-46.
// 327680 columns of 90 levels: the FP64 column solve 3470 / 3710 -> 3314 / 3576
// us (predictor / corrector); diff_cell_update 1081 -> 707, diff_edge_smag
// (with its folded coefficients) 2910 -> 2192.
#pragma once
#include "dfloat.cuh"

namespace icon {

// m in [1, 4) (words mhi, lo) as its leading 24 bits (truncated) plus the next
// 23; sc is the unit of the former, 2^-23 below 2 and 2^-22 from there on
__device__ __forceinline__ float lead24(unsigned mhi, unsigned lo) {
  return __uint_as_float(__funnelshift_l(lo, mhi - 0x38000000u, 3));
}
__device__ __forceinline__ float next23(unsigned lo, float sc) {
  return __fmaf_rn(__uint_as_float(0x3f800000u | ((lo >> 6) & 0x7fffffu)), sc, -sc);
}
// f (normal) plus n units of 2^-52 of its binade, n < 2^34 = hi 2^32 + lo
__device__ __forceinline__ double join(float f, unsigned n_hi, unsigned n_lo) {
  const unsigned u = __float_as_uint(f);
  const unsigned long long b = ((unsigned long long)((u >> 3) + 0x38000000u) << 32 | (u << 29)) +
                               ((unsigned long long)n_hi << 32 | n_lo);
  return __longlong_as_double((long long)b);
}

// 1 / x; NaN for 0, subnormals, magnitudes from 2^1022 on, infinities and NaN
__device__ __forceinline__ double rcp(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned ex = hi & 0x7ff00000u, mhi = (hi & 0x000fffffu) | 0x3ff00000u;
  const float mh = lead24(mhi, lo), ml = next23(lo, 0x1p-23f);
  const float r = fmaxf(__uint_as_float(__float_as_uint(__fdividef(1.0f, mh)) - 8u), 0.5f);
  const float e = __fmaf_rn(-ml, r, __fmaf_rn(-mh, r, 1.0f));       // 1 - m r, in (0, 2^-19)
  const float d = __fmul_rn(r, __fmaf_rn(e, e, e));
  const unsigned n = __float2uint_rn(__fmul_rn(d, 0x1p48f));
  const double y = join(r, n >> 27, n << 5);
  const double m = __hiloint2double((int)mhi, (int)lo);
  const double z = fma(y, fma(-m, y, 1.0), y);
  const unsigned zh = ((unsigned)__double2hiint(z) + 0x3ff00000u - ex) | (hi & 0x80000000u);
  return __hiloint2double(ex - 0x00100000u < 0x7fc00000u ? (int)zh : 0x7ff80000, __double2loint(z));
}

// sqrt(x); zero, subnormals, negative values, infinities and NaN by the library's
__device__ __forceinline__ double sqrt2(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  if (hi - 0x00100000u >= 0x7fe00000u) return sqrt(x);
  const int sh = ((int)(hi >> 20) - 1023) & ~1;
  const unsigned mhi = hi - ((unsigned)sh << 20);
  const float mh = lead24(mhi, lo), ml = next23(lo, mhi >= 0x40000000u ? 0x1p-22f : 0x1p-23f);
  const float q = rsqrtf(mh), h = 0.5f * q;
  const float g = fmaxf(__uint_as_float(__float_as_uint(__fmul_rn(mh, q)) - 16u), 1.0f);
  const float e = __fmul_rn(__fadd_rn(__fmaf_rn(-g, g, mh), ml), h);  // (m - g^2) / 2g, in (0, 2^-18)
  const float d = __fmaf_rn(-__fmul_rn(e, e), h, e);
  const unsigned n = __float2uint_rn(__fmul_rn(d, 0x1p46f));
  const double y = join(g, n >> 26, n << 6);
  const double m = __hiloint2double((int)mhi, (int)lo);
  // 1 / 2y for the correction, to about 2^-42 as well
  const float hb = fmaxf(__uint_as_float(__float_as_uint(h) - 8u), 0.25f);
  const float t = __fmaf_rn(-2.0f * d, hb, __fmaf_rn(-2.0f * g, hb, 1.0f));
  const unsigned nh = __float2uint_rn(__fmul_rn(__fmul_rn(hb, t), 0x1p48f));
  const double z = fma(fma(-y, y, m), join(hb, nh >> 26, nh << 6), y);
  return __hiloint2double(__double2hiint(z) + (sh << 19), __double2loint(z));
}

}  // namespace icon
