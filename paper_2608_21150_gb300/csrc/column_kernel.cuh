// Row A7: vertically implicit solve of w, rho, exner and theta_v, several
// threads per column; only the tridiagonal Thomas sweep, which is sequential in
// the vertical, has one.
//
// Equations (an ICON-type reading; the paper names the solver but gives no
// formula, Sec. 4.1), for full levels k (dz) and interior half levels k (dzh),
// beta the implicit weight, pr = exner - exner_ref, primes the new values:
//   rho'_k = rho_k - dt div_m_k - dt/dz_k [(1-beta)(Fw_k - Fw_k+1) + beta(Fw'_k - Fw'_k+1)],
//   pr'_k  = pr_k - zb_k [dz_k div_t_k + (1-beta)(Gw_k - Gw_k+1) + beta(Gw'_k - Gw'_k+1)],
//   w'_k   = w_k + dt ddt_w_k - dt cpd [theta_ic ((1-beta) dpr_k + beta dpr'_k)/dzh_k
//                                       + theta'_ic dexner_ref_k],
// with Fw = rho_ic w, Gw = rho_ic theta_ic w, zb = dt (rd/cvd) exner/(rho theta dz)
// and w = 0 at the top and the ground.  Eliminating pr' gives a tridiagonal
// system in w'; Thomas elimination top-down, Rayleigh damping, then
// back-substitution.  Arranged for few FP64 operations (the FP64 pipe bounds
// this kernel): with gam_k = dt cpd beta theta_ic/dzh_k, the explicit pressure
// term is gam_k ((1-beta)/beta)(pr_k-1 - pr_k), carried in
// S_k = pr*_k + ((1-beta)/beta) pr_k together with the implicit one; the
// matrix entries use p_k = zb_k A_k and q_k = zb_k A_k+1 (A = beta (rho
// theta)_ic at the half levels); theta_ic is the reference theta at the half
// level plus the interpolated perturbation.  theta'_v from the linearised
// equation of state
//   theta' = theta (rho/rho')(1 + (cvd/rd)(pr' - pr)/exner)
//          = (dt rd/(cvd dz)) (exner - (cvd/rd) pr + (cvd/rd) pr') / (zb rho').
//
// Memory: the state is level-contiguous, so a warp whose lanes are columns
// would read every 32-byte sector for 8 useful bytes.  Instead each CTA stages
// chunks of KC levels (4, 6 or 8, picked by the autotuner for the predictor and
// the corrector) of every input through shared memory with coalesced
// asynchronous copies (a column's chunk is a contiguous run), and stages its
// outputs the same way.  Each chunk's slice of the per-level table is staged
// with them (FP64 or double-word): a warp reads one level of it at a time, with
// 16 columns per CTA two.
// The scratch between the sweeps is laid out so that a thread reaches a
// level's planes from one address and a warp's accesses are coalesced; it is
// written as streaming data and read back evict-first, while the input rows
// are kept (L2 policies below).  The predictor and corrector forms are
// separate kernels.
//
// Measured, predictor / corrector, against one thread walking each column (64
// columns and two warps per CTA, ten warps an SM): R2B2 L30 FP64 98 / 104 ->
// 27 / 27 us, R2B4 L65 FP64 277 / 287 -> 197 / 213 us, R2B6 L90 double-word
// 1.87 / 2.64 -> 1.59 / 2.06 ms, R2B5 L90 double-word over terrain 1.09 / 1.36
// -> 0.70 / 0.94 ms.  R2B6 L90 FP64 3.41 / 3.67 -> 3.31 / 3.58 ms: there both
// keep the FP64 unit busy (a warp's FP64 instruction takes 16 cycles of the SM
// at best and 19 here; 56.9 of them a level in the predictor's chunks of 8, 63.5
// in the corrector's of 4), and only the reciprocal's operations counted.
//
// This header holds the kernel template and its helpers; kernels_column.cu
// instantiates the flat-ground forms (and the allocation-free entry point),
// kernels_column_terrain.cu the terrain-following ones.
#pragma once
#include <cuda_runtime.h>

#include <cmath>
#include <type_traits>

#include "dfloat.cuh"
#include "fp64.cuh"
#include "kernels.h"

namespace icon {
namespace {

// One form of the column solve: CW columns per CTA, chunks of KC levels, RL
// consecutive levels of a chunk per worker thread.  NW worker threads (CW KC /
// RL) and one warp more, which eliminates the last chunk's rows; the warps
// take turns at that.
// Shared memory (bytes): the input tiles of a chunk, [column][KC + 1] with the
// level below the chunk last (a column's levels are contiguous for the copies,
// and the odd row length keeps 32 columns in different banks); then the
// half-level planes [KC + 1][CW] (fr, fg, al, gam, rhs), the matrix rows
// [4][KC][CW], the values carried from chunk to chunk and the chunk's slice of
// the per-level table (16 slots per level).  The back-substitution stages its
// outputs over the tiles and two chunks' w in the first two planes.
template <class T, int KC, int CW, int RL, bool kCorrTiles, bool kTerr>
struct ColForm {
  static constexpr int S = KC / RL;       // worker threads per column
  static constexpr int NW = CW * S;
  static constexpr int kWorkers = NW / 32;
  static constexpr int kWarps = kWorkers + 1;
  static constexpr int NT = 32 * kWarps;
  static constexpr int LD = KC + 1;
  static constexpr int kTile = CW * LD;
  static constexpr int kTiles = (kCorrTiles ? 8 : 6) * kTile;                       // doubles
  static constexpr int kTilesT = ((kCorrTiles ? 2 : 1) + (kTerr ? 1 : 0)) * kTile;  // of type T
  static constexpr int kOut = 4 * kTile * 8 + 3 * kTile * 4;                        // bytes
  static constexpr int kIn = kTiles * 8 + kTilesT * (int)sizeof(T);
  static constexpr int kPlane = (KC + 1) * CW;
  static constexpr int kPlanes0 = ((kIn > kOut ? kIn : kOut) + 15) / 16 * 16;
  static constexpr int kRows0 = kPlanes0 + 5 * kPlane * 8;
  static constexpr int kCarry0 = kRows0 + 4 * KC * CW * 8;
  static constexpr int kLev0 = kCarry0 + 8 * CW * 8;
  static constexpr size_t bytes = (size_t)kLev0 + 16 * (size_t)(KC + 1) * 8;
  // CTAs per SM: the shared-memory limit (233 472 bytes an SM, 1 KB of it
  // reserved per CTA), at most what leaves 80 registers a thread (96 in the
  // narrow form, which small grids run with fewer CTAs than fit)
  static constexpr int by_smem = (int)(233472 / (bytes + 1024));
  static constexpr int by_regs = 65536 / ((CW < 32 ? 96 : 80) * NT);
  static constexpr int blocks = by_smem < 1 || by_regs < 1 ? 1 : (by_smem < by_regs ? by_smem : by_regs);
  static_assert(KC % RL == 0 && NW % 32 == 0 && 32 % CW == 0, "whole runs, whole warps");
};
// Scratch of the solve, [level][group of CW columns][8 planes][CW]: a level's
// planes of one group are neighbours, so a thread reaches all of them from one
// address.  cp, rp: the eliminated rows; rs, ps: the explicit rho, pr; ri, al:
// half-level rho and beta (rho theta); eb, zb: written by the predictor and read
// by the corrector as well.
enum { SCP = 0, SRP = 1, SRS = 2, SPS = 3, SRI = 4, SAL = 5, SEB = 6, SZB = 7 };
constexpr int kScratchPlanes = 8;

// column coefficients: CTHI the reference theta_v at the half level (theta_ic
// is it plus the interpolated perturbation); the explicit part
// of the vertical pressure-gradient term is CGAM (1 - beta)/beta.
enum { CZB = 0, CR = 1, CRN = 2, CTHI = 3, CB = 4, CGAM = 5, WG = 6, WG2 = 7 };

// 8-byte asynchronous global->shared copy (no register staging), completed
// by cp_wait() for all copies the thread issued.
__device__ __forceinline__ void cp8(double* dst, const double* src) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(src) : "memory");
}
// The row-gathered input copies mark their lines evict-last in L2: a chunk
// reads a few levels of every row, so the rest of a 128-byte line is used
// by the next chunks of the same CTA, and the Thomas scratch streaming
// through L2 meanwhile should be evicted first.
__device__ __forceinline__ unsigned long long policy_evict_last() {
  unsigned long long p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;\n" : "=l"(p));
  return p;
}
__device__ __forceinline__ void cp_async(double* dst, const double* src, unsigned long long pol) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global.L2::cache_hint [%0], [%1], 8, %2;\n" ::"r"(s), "l"(src), "l"(pol) : "memory");
}
__device__ __forceinline__ void cp_async(float* dst, const float* src, unsigned long long pol) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global.L2::cache_hint [%0], [%1], 4, %2;\n" ::"r"(s), "l"(src), "l"(pol) : "memory");
}
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// tile[col][kk] = X[row(col) * ld + k0 + kk] for kk < nk: consecutive worker
// threads (wt) copy consecutive levels of one row; off[j] = row * ld + kk of the
// thread's j-th copy.
template <class F, int KC, class X>
__device__ __forceinline__ void tile_rows(X* tile, const X* __restrict__ src, int wt, const size_t* off, int k0,
                                          int nk, unsigned long long pol) {
#pragma unroll
  for (int j = 0; j < KC / F::S; ++j) {
    const int i = wt + j * F::NW;
    const int col = i / KC, kk = i - col * KC;
    if (kk < nk) cp_async(tile + col * F::LD + kk, src + off[j] + k0, pol);
  }
}
// rows [col][kk] of a staged output tile back to X[(c0 + col) * ld + k0 + kk]
template <class F, int KC, class X>
__device__ __forceinline__ void store_rows(const X* tile, X* __restrict__ dst, int wt, const size_t* off, int k0,
                                           int nk, int ncol) {
#pragma unroll
  for (int j = 0; j < KC / F::S; ++j) {
    const int i = wt + j * F::NW;
    const int col = i / KC, kk = i - col * KC;
    if (kk < nk && col < ncol) dst[off[j] + k0] = tile[col * F::LD + kk];
  }
}

template <class T>
struct ColArgs {
  const double *w, *rho, *exner, *theta, *rho_p, *theta_p, *div_m, *div_t;
  const T *ddt_w0, *ddt_w1;
  double *col, *w_o, *rho_o, *exner_o, *theta_o;
  // mixed mode: FP32 mirrors of the outputs (w; rho, theta_v perturbations)
  float *m_w, *m_rho, *m_th;
  // terrain: contravariant correction of the winds (cells, half levels)
  const T* wcc;
  // row stride of the fields of type T and of the mirrors
  int ldt;
};

// Arithmetic of the solve: FP64 (R = double), or double-word FP32 (R = dws,
// mixed precision) with inputs split and outputs joined at the tile boundary.
// mad is a b + c: one FP64 instruction, written out so that every form of
// the kernel rounds alike, or the double-word product and sum; mul is a product
// that must not be fused with the sum it feeds.
template <class R>
struct Ar;
template <>
struct Ar<double> {
  static __device__ __forceinline__ double in(double x) { return x; }
  static __device__ __forceinline__ double in(float x) { return (double)x; }
  static __device__ __forceinline__ double inv(double x) { return rcp(x); }
  static __device__ __forceinline__ double out(double x) { return x; }
  static __device__ __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }
  static __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
};
template <>
struct Ar<dws> {
  static __device__ __forceinline__ dws in(double x) { return to_dws(to_df(x)); }
  static __device__ __forceinline__ dws in(float x) { return {x, 0.0f}; }
  static __device__ __forceinline__ dws inv(dws x) { return rcp(x); }
  static __device__ __forceinline__ double out(dws x) { return to_double(x); }
  static __device__ __forceinline__ dws mad(dws a, dws b, dws c) { return a * b + c; }
  static __device__ __forceinline__ dws mul(dws a, dws b) { return a * b; }
};

// per-level quantities: j < 8 the column coefficients, then these
enum { LEX = 8, LTH = 9, LDZ = 10, LRAY = 11, LRHO = 12 };
template <class R, int J>
__device__ __forceinline__ R lev(const DevVert& v, int k);
template <>
__device__ __forceinline__ double lev<double, LEX>(const DevVert& v, int k) { return v.exner_ref[k]; }
template <>
__device__ __forceinline__ double lev<double, LTH>(const DevVert& v, int k) { return v.theta_ref[k]; }
template <>
__device__ __forceinline__ double lev<double, LDZ>(const DevVert& v, int k) { return v.dz[k]; }
template <>
__device__ __forceinline__ double lev<double, LRAY>(const DevVert& v, int k) { return v.ray_fac[k]; }
template <class R, int J>
__device__ __forceinline__ R lev(const DevVert& v, int k) {
  if constexpr (!std::is_same<R, double>::value) {
    return reinterpret_cast<const R*>(v.lev_hl)[16 * (size_t)k + J];
  } else {
    static_assert(J < 8, "column coefficient");
    return v.colc[8 * (size_t)k + J];
  }
}

// Per-level quantity of level k: from the chunk's copy of the table in shared
// memory (Ls: levels from k0 on, 16 slots each; kStaged), else from the
// device arrays.
template <class R, int J, bool kStaged>
__device__ __forceinline__ R levs(const DevVert& v, const double* Ls, int k, int k0) {
  if constexpr (kStaged) {
    return *reinterpret_cast<const R*>(Ls + 16 * (k - k0) + J);
  } else {
    return lev<R, J>(v, k);
  }
}

// Per-level quantity J of level k: over terrain (kTerr) this column's own
// value from the slot-major, level-major table v.colt, else levs.
template <class R, int J, bool kStaged, bool kTerr>
__device__ __forceinline__ R levc(const DevVert& v, const double* Ls, int k, int k0, int c, int nc) {
  if constexpr (kTerr) {
    return *reinterpret_cast<const R*>(v.colt + ((size_t)J * (v.nlev + 1) + k) * nc + c);
  } else {
    return levs<R, J, kStaged>(v, Ls, k, k0);
  }
}

// FP32 mirror value of a solve result: the double-word pair's leading sum,
// or the FP64 value narrowed without the FP64 pipe
__device__ __forceinline__ float mirror_f32(dws x) { return to_float(x); }
__device__ __forceinline__ float mirror_f32(double x) { return to_float(to_df(x)); }

// x - q for the terrain's contravariant correction q (type T).  In FP64 a
// plain subtraction (exact where q = 0).  In double-word arithmetic x itself
// where q is exactly zero, so that the pairs the FP64 inputs are split into (a
// truncated leading word) are not renormalised over flat ground: equal
// columns then step like the flat dycore bit for bit in either arithmetic.
// (A select in the FP64 form changes how the compiler fuses the products of
// x into multiply-adds, and with it the last bit.)
template <class R, class T>
__device__ __forceinline__ R minus_corr(R x, T q) {
  if constexpr (std::is_same<R, double>::value) {
    return x - Ar<R>::in(q);
  } else {
    return q == T(0) ? x : x - Ar<R>::in(q);
  }
}

// A value the mixed-precision step (T = float) keeps as a double-word pair in
// an 8-byte slot -- the flux divergences and the predictor's rho and theta_v
// -- read as the pair; otherwise an FP64 value, converted.
template <class T, class R>
__device__ __forceinline__ R stored_in(const double* p) {
  if constexpr (std::is_same<T, float>::value && !std::is_same<R, double>::value) {
    return *reinterpret_cast<const R*>(p);
  } else {
    return Ar<R>::in(*p);
  }
}

// A horizontal flux divergence: the mixed-precision stencils (T = float)
// store it as a double-word pair in its 8-byte slot whatever the solve's
// arithmetic R (read as the pair, or widened to FP64 exactly); else FP64.
template <class T, class R>
__device__ __forceinline__ R stored_div(const double* p) {
  if constexpr (std::is_same<T, float>::value) {
    const df x = *reinterpret_cast<const df*>(p);
    if constexpr (std::is_same<R, double>::value) {
      return f2d_exact(x.hi) + f2d_exact(x.lo);
    } else {
      return to_dws(x);
    }
  } else {
    return Ar<R>::in(*p);
  }
}

// Scratch planes hold R values in 8-byte slots (a double-word value is two floats).  They
// are read back only after the whole forward sweep, so they are stored as
// streaming (evict-first) data that does not displace the input rows in L2.
__device__ __forceinline__ void put(double* p, double x) { __stcs(p, x); }
__device__ __forceinline__ void put(double* p, dws x) { __stcs(reinterpret_cast<float2*>(p), make_float2(x.hi, x.lo)); }
template <class R>
__device__ __forceinline__ R get(const double* p) {
  return *reinterpret_cast<const R*>(p);
}
// a scratch value read for the last time (evict-first)
template <class R>
__device__ __forceinline__ R get_last(const double* p) {
  if constexpr (std::is_same<R, double>::value) {
    return __ldcs(p);
  } else {
    const float2 x = __ldcs(reinterpret_cast<const float2*>(p));
    return {x.x, x.y};
  }
}

// Barrier of the worker threads alone (barrier 0 is the whole CTA's).
template <class F>
__device__ __forceinline__ void sync_workers() {
  asm volatile("bar.sync 1, %0;\n" ::"n"(F::NW) : "memory");
}

// The solve, CW columns per CTA and S = KC / RL threads per column: thread
// (col, sub) owns RL consecutive levels of every chunk of KC.  Only the
// elimination and the substitution are sequential in the vertical; the rest
// of a chunk is done by all threads at once:
//   half levels  interpolated state, explicit fluxes, row factors gam, rhs
//   levels       zb, the explicit parts rho*, pr*, and p, q, S
//   rows         the matrix rows from two neighbouring levels
//   elimination  one thread per column, in a warp that works on the last
//                chunk's rows while the others are at the next (the warps take
//                turns, so that no scheduler of the SM has all the chains)
// with what a neighbour needs passed through shared memory.  One FP64
// instruction of a warp occupies its scheduler's FP64 unit for 64 cycles
// whatever its active lanes, so a column walked by one thread takes 60 x 64
// cycles a level and a grid of a few thousand columns leaves most schedulers
// idle: that bounded the grids up to R2B5, the double-word form's ten warps
// an SM bounded the large ones.
//
// kOwnZb: the corrector form computes zb and the equation-of-state term itself
// (as the predictor does) instead of reading the predictor's; used by the
// allocation-free entry point.
// kCorr: 0 the predictor form, 1 the corrector form, -1 the form the
// `corrector` argument names (one kernel for both; the allocation-free entry).
// kTerr: per-column metrics and the solve in the contravariant velocity
// w - wcc (zero at the top and the ground, where w = wcc: the kinematic
// ground condition); the fluxes rho_ic w and the Rayleigh damping act on it.
template <class T, class R, int KC, int CW, int RL, int kCorr, bool kTerr, bool kOwnZb>
__global__ void __launch_bounds__(ColForm<T, KC, CW, RL, kCorr != 0, kTerr>::NT,
                                  ColForm<T, KC, CW, RL, kCorr != 0, kTerr>::blocks)
    sn_column(int nc, DevVert v, Scalars sc, int corrector_arg, ColArgs<T> a) {
  using F = ColForm<T, KC, CW, RL, kCorr != 0, kTerr>;
  using A = Ar<R>;
  const bool corrector = kCorr < 0 ? corrector_arg != 0 : kCorr == 1;
  constexpr bool kDW = !std::is_same<R, double>::value;
  // the mixed step's engine path (FP32 stencil inputs, double-word solve)
  constexpr bool kPairs = std::is_same<T, float>::value && kDW;
  // FP32 stencils read FP32 mirrors of the solve's outputs (either arithmetic)
  constexpr bool kMirror = std::is_same<T, float>::value;
  constexpr bool kCT = kCorr != 0;
  constexpr int LD = F::LD;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  double* sm = reinterpret_cast<double*>(sm_raw);
  const unsigned tid = after_previous(threadIdx.x);
  const int lane = tid & 31, warp = tid >> 5;
  const int col = lane % CW;
  const int nlev = v.nlev, nlevp = nlev + 1;
  const int c0 = blockIdx.x * CW;
  const bool active = c0 + col < nc;
  const int c = min(c0 + col, nc - 1);  // spare threads walk the last column and store nothing
  const int ncol = min(CW, nc - c0);
  // step i of a sweep: the warps take turns at the elimination; the others
  // are the workers 0 .. kWorkers - 1 of the step
  auto role = [&](int i) { return (warp + (int)((blockIdx.x + i) % F::kWarps)) % F::kWarps; };

  double* T_w = sm;
  double* T_rho = T_w + F::kTile;
  double* T_th = T_rho + F::kTile;
  double* T_rp = T_th + F::kTile;                       // corrector
  double* T_tp = T_rp + F::kTile;                       // corrector
  double* T_pi = T_th + (kCT ? 3 : 1) * F::kTile;       // then S
  double* T_dm = T_pi + F::kTile;                       // then p
  double* T_dt = T_dm + F::kTile;                       // then q
  T* T_dw0 = reinterpret_cast<T*>(T_dt + F::kTile);     // tendencies at the half level below
  T* T_dw1 = T_dw0 + F::kTile;                          // corrector
  T* T_wc = T_dw0 + (kCT ? 2 : 1) * F::kTile;           // terrain: contravariant correction, half level below
  // planes: row kk is the half level above level k0 + kk
  R* P_fr = reinterpret_cast<R*>(sm_raw + F::kPlanes0);
  R* P_fg = P_fr + F::kPlane;
  R* P_al = P_fg + F::kPlane;
  R* P_gm = P_al + F::kPlane;
  R* P_rh = P_gm + F::kPlane;
  // the matrix rows of a chunk: gam p_k-1, gam q_k, the diagonal, the right-hand side
  R* M_gp = reinterpret_cast<R*>(sm_raw + F::kRows0);
  R* M_gq = M_gp + KC * CW;
  R* M_d = M_gq + KC * CW;
  R* M_r = M_d + KC * CW;
  R* K_pqs = reinterpret_cast<R*>(sm_raw + F::kCarry0);  // [2][3][CW]: p, q, S of the last chunk's last level
  R* K_el = K_pqs + 6 * CW;                              // [2][CW]: the elimination's (and substitution's) state
  // the per-level table is staged per chunk, except in the FP64 form of the
  // allocation-free entry, which has no FP64 copy of the table
  // (over terrain only for the FP32 mirrors' offsets of the mixed modes;
  // every physical quantity is the column's own)
  constexpr bool kStage = kTerr ? (kDW || kMirror) : (kDW || !kOwnZb);
  double* L_s = reinterpret_cast<double*>(sm_raw + F::kLev0);
  const double* lev_src = kDW ? reinterpret_cast<const double*>(v.lev_hl) : v.lev64;

  const size_t s_lev = (size_t)gridDim.x * kScratchPlanes * CW;  // scratch: one level
  double* s_col = a.col + (size_t)blockIdx.x * kScratchPlanes * CW + col;

  const R zero = A::in(0.0), one = A::in(1.0);
  const R dt = A::in(sc.dt_s), beta = A::in(sc.beta), ombeta = A::in(1.0 - sc.beta);
  const R wn_r = A::in(sc.wnow_rth), wnew_r = A::in(sc.wnew_rth);
  const R dt_wn_v = A::in(sc.dt_s * sc.wnow_vel), dt_wnew_v = A::in(sc.dt_s * sc.wnew_vel);
  const R cvd_o_rd = A::in(sc.cvd_o_rd), ex_o_im = A::in((1.0 - sc.beta) / sc.beta);
  const float wn_vf = to_float(to_df(sc.wnow_vel)), wnew_vf = to_float(to_df(sc.wnew_vel));
  // levels k < n_ray may be Rayleigh-damped (the factor is 1 below)
  const int n_ray = v.n_ray;

  // element offsets of worker wt's copies (FP64 full and half levels, type T)
  auto offsets = [&](int wt, size_t* of, size_t* oh, size_t* ot) {
#pragma unroll
    for (int j = 0; j < RL; ++j) {
      const int i = wt + j * F::NW;
      const size_t r = min(c0 + i / KC, nc - 1);
      of[j] = r * nlev + i % KC;
      oh[j] = r * nlevp + i % KC;
      ot[j] = r * a.ldt + i % KC;
    }
  };
  const unsigned long long pol = policy_evict_last();
  auto load_chunk = [&](int k0, int wt) {
    const int nk = min(KC, nlev - k0);
    size_t of[RL], oh[RL], ot[RL];
    offsets(wt, of, oh, ot);
    tile_rows<F, KC>(T_w, a.w, wt, oh, k0, nk, pol);
    tile_rows<F, KC>(T_rho, a.rho, wt, of, k0, nk, pol);
    tile_rows<F, KC>(T_th, a.theta, wt, of, k0, nk, pol);
    tile_rows<F, KC>(T_pi, a.exner, wt, of, k0, nk, pol);
    tile_rows<F, KC>(T_dm, a.div_m, wt, of, k0, nk, pol);
    tile_rows<F, KC>(T_dt, a.div_t, wt, of, k0, nk, pol);
    tile_rows<F, KC>(T_dw0, a.ddt_w0, wt, ot, k0 + 1, nk, pol);
    if constexpr (kTerr) tile_rows<F, KC>(T_wc, a.wcc, wt, ot, k0 + 1, nk, pol);
    if (kCT && corrector) {
      tile_rows<F, KC>(T_dw1, a.ddt_w1, wt, ot, k0 + 1, nk, pol);
      tile_rows<F, KC>(T_rp, a.rho_p, wt, of, k0, nk, pol);
      tile_rows<F, KC>(T_tp, a.theta_p, wt, of, k0, nk, pol);
    }
    // the level below the chunk
    if (wt < CW) {
      const int o = col * LD + nk;
      cp_async(T_w + o, a.w + (size_t)c * nlevp + k0 + nk, pol);
      if (k0 + nk < nlev) {
        const size_t i = (size_t)c * nlev + k0 + nk;
        cp_async(T_rho + o, a.rho + i, pol);
        cp_async(T_th + o, a.theta + i, pol);
        if (kCT && corrector) {
          cp_async(T_rp + o, a.rho_p + i, pol);
          cp_async(T_tp + o, a.theta_p + i, pol);
        }
      }
    }
    if constexpr (kStage) {
      for (int i = wt; i < 16 * min(KC + 1, nlev - k0); i += F::NW) cp8(L_s + i, lev_src + 16 * (size_t)k0 + i);
    }
  };

  // double-word code is long: its loops stay rolled, for the instruction cache
  constexpr int kUnroll = kDW ? 1 : RL;
  const int nch = (nlev + KC - 1) / KC;
  if (role(0) < F::kWorkers) load_chunk(0, role(0) * 32 + lane);
#pragma unroll 1
  for (int ch = 0; ch <= nch; ++ch) {
    const int k0 = ch * KC, nk = min(KC, nlev - k0);
    const int r = role(ch), sub = (r * 32 + lane) / CW;
    const bool work = r < F::kWorkers && ch < nch;
    if (work) {
      // the predictor's zb of this thread's levels, in flight until the levels are at hand
      R zb_in[RL];
      if (kCT && corrector && !kOwnZb) {
#pragma unroll
        for (int j = 0; j < RL; ++j) {
          const int kk = sub * RL + j;
          zb_in[j] = kk < nk ? get<R>(s_col + (size_t)(k0 + kk) * s_lev + SZB * CW) : zero;
        }
      }
      cp_wait();
      sync_workers<F>();
      // ---- half levels: row kk + 1 is the half level below level k0 + kk
      if (ch == 0 && sub == 0) {  // row 0: the top, then carried from chunk to chunk
        const R w0 = A::in(T_w[col * LD]);
        P_fr[col] = zero * w0;
        P_fg[col] = zero * w0;
        P_al[col] = zero;
      }
      R ra_c = zero, tpa_c = zero;
#pragma unroll kUnroll
      for (int j = 0; j <= RL; ++j) {
        // pass j: the levels' averages at k, then (from the second pass on) the half level k
        const int kk = sub * RL + j, k = k0 + kk;
        if (kk > nk) break;
        const int o = col * LD + kk;
        R ra_x = zero, tpa_x = zero;
        const bool inside = k < nlev;
        if (inside) {
          ra_x = A::in(T_rho[o]);
          R ta = A::in(T_th[o]);
          if (corrector) {  // time averages
            ra_x = A::mad(wn_r, ra_x, wnew_r * stored_in<T, R>(T_rp + o));
            ta = A::mad(wn_r, ta, wnew_r * stored_in<T, R>(T_tp + o));
          }
          tpa_x = ta - levc<R, LTH, kStage, kTerr>(v, L_s, k, k0, c, nc);
        }
        if (j > 0) {
          R ric = zero, tic = zero, tpic = zero;
          if (inside) {
            const R g1 = levc<R, WG, kStage, kTerr>(v, L_s, k, k0, c, nc);
            const R g2 = levc<R, WG2, kStage, kTerr>(v, L_s, k, k0, c, nc);
            ric = A::mad(g1, ra_c, g2 * ra_x);
            // the perturbation interpolated from the levels' perturbations (no
            // cancellation against the reference), the total from it
            tpic = A::mad(g1, tpa_c, g2 * tpa_x);
            tic = levc<R, CTHI, kStage, kTerr>(v, L_s, k, k0, c, nc) + tpic;
          }
          const R w1 = A::in(T_w[o]);
          const T wcc = kTerr ? T_wc[o - 1] : T(0);
          const R wf = kTerr ? minus_corr(w1, wcc) : w1;
          const R rt = ric * tic;
          const R al = beta * rt;
          const int q = kk * CW + col;
          P_fr[q] = ric * wf;
          P_fg[q] = rt * wf;
          P_al[q] = al;
          if (inside) {
            // w + dt (time-averaged tendency)
            R w0;
            if constexpr (std::is_same<T, float>::value) {  // FP32 tendencies: their time average in FP32
              w0 = A::mad(dt, A::in(corrector ? fmaf(wn_vf, T_dw0[o - 1], wnew_vf * T_dw1[o - 1]) : T_dw0[o - 1]),
                          w1);
            } else {
              w0 = corrector ? A::mad(dt_wnew_v, A::in(T_dw1[o - 1]), A::mad(dt_wn_v, A::in(T_dw0[o - 1]), w1))
                             : A::mad(dt, A::in(T_dw0[o - 1]), w1);
            }
            P_gm[q] = levc<R, CGAM, kStage, kTerr>(v, L_s, k, k0, c, nc) * tic;
            P_rh[q] = A::mad(-levc<R, CB, kStage, kTerr>(v, L_s, k, k0, c, nc), tpic,
                             kTerr ? minus_corr(w0, wcc) : w0);
            if (active) {
              double* sp = s_col + (size_t)k * s_lev;
              put(sp + SRI * CW, ric);
              put(sp + SAL * CW, al);
            }
          }
        }
        ra_c = ra_x;
        tpa_c = tpa_x;
      }
      sync_workers<F>();
      // ---- levels: explicit parts, and p, q, S over the consumed tiles
#pragma unroll kUnroll
      for (int j = 0; j < RL; ++j) {
        const int kk = sub * RL + j, k = k0 + kk;
        if (kk >= nk) break;
        const int o = col * LD + kk, q = kk * CW + col;
        double* sp = s_col + (size_t)k * s_lev;
        R zb = zero;
        if (kCT && corrector && !kOwnZb) {
#pragma unroll
          for (int i = 0; i < RL; ++i)
            if (i == j) zb = zb_in[i];
        }
        const R rho_n = A::in(T_rho[o]), pi_n = A::in(T_pi[o]);
        const R pr = pi_n - levc<R, LEX, kStage, kTerr>(v, L_s, k, k0, c, nc);
        if (!corrector || kOwnZb) {
          zb = levc<R, CZB, kStage, kTerr>(v, L_s, k, k0, c, nc) * pi_n * A::inv(rho_n * A::in(T_th[o]));
          if (active) {
            put(sp + SZB * CW, zb);
            put(sp + SEB * CW, A::mad(-cvd_o_rd, pr, pi_n));
          }
        }
        const R rstar = A::mad(-levc<R, CR, kStage, kTerr>(v, L_s, k, k0, c, nc), P_fr[q] - P_fr[q + CW],
                               A::mad(-dt, stored_div<T, R>(T_dm + o), rho_n));
        const R pstar = A::mad(-zb, A::mad(ombeta, P_fg[q] - P_fg[q + CW],
                                           levc<R, LDZ, kStage, kTerr>(v, L_s, k, k0, c, nc) * stored_div<T, R>(T_dt + o)),
                               pr);
        if (active) {
          put(sp + SRS * CW, rstar);
          put(sp + SPS * CW, pstar);
        }
        *reinterpret_cast<R*>(T_dm + o) = zb * P_al[q];
        *reinterpret_cast<R*>(T_dt + o) = zb * P_al[q + CW];
        *reinterpret_cast<R*>(T_pi + o) = A::mad(ex_o_im, pr, pstar);
      }
    } else if (r == F::kWorkers && ch > 0) {
      // ---- elimination of the last chunk's rows
      const int ke = k0 - KC;
      R cp = ke == 0 ? zero : K_el[col], rp = ke == 0 ? zero : K_el[CW + col];
#pragma unroll 1
      for (int kk = ke == 0 ? 1 : 0; kk < min(KC, nlev - ke); ++kk) {
        const int q = kk * CW + col;
        const R gp = M_gp[q];
        const R inv = A::inv(A::mad(gp, cp, M_d[q]));
        rp = A::mad(gp, rp, M_r[q]) * inv;
        cp = -M_gq[q] * inv;
        if (active && lane < CW) {
          double* sp = s_col + (size_t)(ke + kk) * s_lev;
          put(sp + SCP * CW, cp);
          put(sp + SRP * CW, rp);
        }
      }
      __syncwarp();
      if (lane < CW) {
        K_el[col] = cp;
        K_el[CW + col] = rp;
      }
    }
    if (ch == nch) break;
    __syncthreads();  // the levels are done, and the elimination with the last chunk's rows
    if (work) {
      // ---- rows: -gam p_k-1 w'_k-1 + (1 + gam (q_k-1 + p_k)) w'_k - gam q_k w'_k+1 = rm
#pragma unroll kUnroll
      for (int j = 0; j < RL; ++j) {
        const int kk = sub * RL + j;
        if (kk >= nk) break;
        const int o = col * LD + kk, q = kk * CW + col;
        const R p = get<R>(T_dm + o), qq = get<R>(T_dt + o), s = get<R>(T_pi + o);
        if (k0 + kk >= 1) {
          R pm, qm, smn;
          if (kk == 0) {
            const R* kp = K_pqs + ((ch + 1) & 1) * 3 * CW + col;
            pm = kp[0];
            qm = kp[CW];
            smn = kp[2 * CW];
          } else {
            pm = get<R>(T_dm + o - 1);
            qm = get<R>(T_dt + o - 1);
            smn = get<R>(T_pi + o - 1);
          }
          const R gam = P_gm[q];
          M_r[q] = A::mad(-gam, smn - s, P_rh[q]);
          M_d[q] = A::mad(gam, qm + p, one);
          M_gp[q] = gam * pm;
          M_gq[q] = gam * qq;
        }
        if (kk == nk - 1) {  // for the next chunk
          R* kp = K_pqs + (ch & 1) * 3 * CW + col;
          kp[0] = p;
          kp[CW] = qq;
          kp[2 * CW] = s;
        }
        if (kk == 0) {  // the half level below the chunk becomes row 0
          const int q1 = nk * CW + col;
          P_fr[q] = P_fr[q1];
          P_fg[q] = P_fg[q1];
          P_al[q] = P_al[q1];
          P_gm[q] = P_gm[q1];
          P_rh[q] = P_rh[q1];
        }
      }
    }
    __syncthreads();  // the rows are ready, the tiles consumed
    if (ch + 1 < nch && role(ch + 1) < F::kWorkers) load_chunk(k0 + KC, role(ch + 1) * 32 + lane);
  }

  // back-substitution over the same chunks, bottom to top: one warp finds w'
  // of a chunk's levels, the others update the levels of the chunk below.  The
  // scratch they read was written by threads of this CTA.
  __syncthreads();
  R* W0 = P_fr;  // [2][KC + 1][CW], row kk: damped w' at the half level above level k0 + kk
  double* O_w = sm;
  double* O_rho = O_w + F::kTile;
  double* O_pi = O_rho + F::kTile;
  double* O_th = O_pi + F::kTile;
  float* Q_w = reinterpret_cast<float*>(O_th + F::kTile);
  float* Q_rho = Q_w + F::kTile;
  float* Q_th = Q_rho + F::kTile;
  // what a level reads of the scratch (ri, al: its upper half level)
  struct Level {
    R ri, al, rs, ps, eb, zb;
  };
  auto read_level = [&](int k, bool in) {
    const double* sp = s_col + (size_t)k * s_lev;
    Level x;
    const bool hl = in && k >= 1;
    x.ri = hl ? get_last<R>(sp + SRI * CW) : zero;
    x.al = hl ? get_last<R>(sp + SAL * CW) : zero;
    x.rs = in ? get_last<R>(sp + SRS * CW) : zero;
    x.ps = in ? get_last<R>(sp + SPS * CW) : zero;
    x.eb = in ? get_last<R>(sp + SEB * CW) : zero;
    x.zb = in ? get<R>(sp + SZB * CW) : one;
    return x;
  };
#pragma unroll 1
  for (int ch = 0; ch <= nch; ++ch) {
    const int r = role(ch);
    if (r == F::kWorkers && ch < nch) {
      const int k0 = (nch - 1 - ch) * KC, nk = min(KC, nlev - k0);
      R* W = W0 + (ch & 1) * F::kPlane;
      R cpv[KC], rpv[KC];
#pragma unroll
      for (int kk = 0; kk < KC; ++kk) {
        const double* sp = s_col + (size_t)(k0 + kk) * s_lev;
        const bool in = kk < nk && k0 + kk >= 1;
        cpv[kk] = in ? get_last<R>(sp + SCP * CW) : zero;
        rpv[kk] = in ? get_last<R>(sp + SRP * CW) : zero;
      }
      R w = ch == 0 ? zero : K_el[col], wd = ch == 0 ? zero : K_el[CW + col];
      W[nk * CW + col] = wd;
#pragma unroll
      for (int kk = KC - 1; kk >= 0; --kk) {
        const int k = k0 + kk;
        if (kk >= nk) continue;
        w = k >= 1 ? A::mad(-cpv[kk], w, rpv[kk]) : zero;
        wd = w;
        if (k >= 1 && k < n_ray) wd = w * levc<R, LRAY, false, kTerr>(v, L_s, k, k0, c, nc);
        W[kk * CW + col] = wd;
      }
      __syncwarp();
      K_el[col] = w;
      K_el[CW + col] = wd;
    } else if (r < F::kWorkers && ch > 0) {
      const int k0 = (nch - ch) * KC, nk = min(KC, nlev - k0);
      const R* W = W0 + ((ch + 1) & 1) * F::kPlane;
      const int wt = r * 32 + lane, sub = wt / CW;
      const int kb = min(sub * RL + RL, nk) - 1;  // this thread's lowest level in the chunk (below sub * RL: none)
      const bool some = kb >= sub * RL;
      Level x = read_level(k0 + kb, some);
      R ri1 = zero, al1 = zero;
      if (some && k0 + kb + 1 < nlev) {
        const double* sp = s_col + (size_t)(k0 + kb + 1) * s_lev;
        ri1 = get<R>(sp + SRI * CW);
        al1 = get<R>(sp + SAL * CW);
      }
      if constexpr (kStage) {
        for (int i = wt; i < 16 * nk; i += F::NW) cp8(L_s + i, lev_src + 16 * (size_t)k0 + i);
        cp_wait();
        sync_workers<F>();
      }
      if (some) {
        const R w1 = W[(kb + 1) * CW + col];
        R fr1 = A::mul(ri1, w1), fa1 = A::mul(al1, w1);
#pragma unroll kUnroll
        for (int kk = kb; kk >= sub * RL; --kk) {
          const int k = k0 + kk, o = col * LD + kk;
          const Level y = x;
          if (kk > sub * RL) x = read_level(k - 1, true);
          const R wd = W[kk * CW + col];
          const R fr = A::mul(y.ri, wd), fa = A::mul(y.al, wd);
          const R rnew = A::mad(-levc<R, CRN, kStage, kTerr>(v, L_s, k, k0, c, nc), fr - fr1, y.rs);
          const R prnew = A::mad(-y.zb, fa - fa1, y.ps);
          const R thnew = levc<R, CZB, kStage, kTerr>(v, L_s, k, k0, c, nc) * A::mad(cvd_o_rd, prnew, y.eb) *
                          A::inv(y.zb * rnew);
          R wt = wd;
          if constexpr (kTerr) wt = minus_corr(wd, -a.wcc[(size_t)c * a.ldt + k]);  // w = w_con + wcc
          if (!(kMirror && !corrector)) O_w[o] = A::out(wt);
          if (kPairs && !corrector) {
            // the mixed predictor's rho and theta_v stay double-word pairs (read by the corrector)
            *reinterpret_cast<R*>(O_rho + o) = rnew;
            *reinterpret_cast<R*>(O_th + o) = thnew;
          } else {
            O_rho[o] = A::out(rnew);
            O_th[o] = A::out(thnew);
          }
          if (a.exner_o) O_pi[o] = A::out(levc<R, LEX, kStage, kTerr>(v, L_s, k, k0, c, nc) + prnew);
          if constexpr (kMirror) {
            Q_w[o] = mirror_f32(wt);
            if (corrector) {
              Q_rho[o] = mirror_f32(rnew - levs<R, LRHO, kStage>(v, L_s, k, k0));
              Q_th[o] = mirror_f32(thnew - levs<R, LTH, kStage>(v, L_s, k, k0));
            }
          }
          fr1 = fr;
          fa1 = fa;
        }
      }
      sync_workers<F>();
      size_t of[RL], oh[RL], ot[RL];
      offsets(wt, of, oh, ot);
      if (a.w_o) store_rows<F, KC>(O_w, a.w_o, wt, oh, k0, nk, ncol);
      store_rows<F, KC>(O_rho, a.rho_o, wt, of, k0, nk, ncol);
      if (a.exner_o) store_rows<F, KC>(O_pi, a.exner_o, wt, of, k0, nk, ncol);
      store_rows<F, KC>(O_th, a.theta_o, wt, of, k0, nk, ncol);
      if constexpr (kMirror) {
        if (a.m_w) store_rows<F, KC>(Q_w, a.m_w, wt, ot, k0, nk, ncol);
        if (a.m_rho) {
          store_rows<F, KC>(Q_rho, a.m_rho, wt, ot, k0, nk, ncol);
          store_rows<F, KC>(Q_th, a.m_th, wt, ot, k0, nk, ncol);
        }
      }
    }
    if (ch < nch) __syncthreads();
  }
  if (active && threadIdx.x < CW) {
    // the ground: w_con = 0, so w = wcc there (0 over flat ground)
    const T wg = kTerr ? a.wcc[(size_t)c * a.ldt + nlev] : T(0);
    if (a.w_o) a.w_o[(size_t)c * nlevp + nlev] = (double)wg;
    if (a.m_w) a.m_w[(size_t)c * a.ldt + nlev] = (float)wg;
  }
}

// Mixed precision (FP32 stencil inputs) solves in double-word FP32 arithmetic;
// the FP64 mode in FP64.
template <class T>
using ColArith = typename std::conditional<std::is_same<T, float>::value, dws, double>::type;

// Arguments of the engine's predictor (corrector = 0: the predicted state
// into the work arrays) or corrector (the new state over st) column solve.
template <class T>
ColArgs<T> col_args(const Engine& en, int corrector, const StateView& st, const T* ddt_w0, const T* ddt_w1) {
  const DevWork& wk = en.wk;
  ColArgs<T> a{};
  a.w = st.w;
  a.rho = st.rho;
  a.exner = st.exner;
  a.theta = st.theta_v;
  a.ddt_w0 = ddt_w0;
  a.ddt_w1 = ddt_w1;
  a.rho_p = wk.rho_p;
  a.theta_p = wk.theta_p;
  a.div_m = wk.div_m;
  a.div_t = wk.div_t;
  a.col = wk.col;
  a.ldt = std::is_same<T, float>::value ? en.c32.v.ldh : en.c64.v.ldh;
  constexpr bool mixed = std::is_same<T, float>::value;
  if (corrector) {
    a.w_o = st.w;
    a.rho_o = st.rho;
    a.exner_o = st.exner;
    a.theta_o = st.theta_v;
    if (mixed) {
      a.m_w = en.m.w;
      a.m_rho = en.m.rho;
      a.m_th = en.m.th;
    }
  } else {
    a.w_o = mixed ? nullptr : wk.w_p;  // mixed: the predicted w is read only as its FP32 mirror
    a.rho_o = wk.rho_p;
    a.exner_o = nullptr;  // the predicted exner has no reader
    a.theta_o = wk.theta_p;
    if (mixed) a.m_w = en.m.w_p;
  }
  return a;
}


// Runs f on a compile-time form of the solve: the narrow one, or the wide ones
// with chunks of 4, 6 or 8 levels.
template <class Fn>
void with_col_form(int kc, bool narrow, Fn&& f) {
  using std::integral_constant;
  if (narrow)
    f(integral_constant<int, 8>{}, integral_constant<int, kColNarrow>{}, integral_constant<int, 1>{});
  else if (kc == 4)
    f(integral_constant<int, 4>{}, integral_constant<int, kColWide>{}, integral_constant<int, 1>{});
  else if (kc == 6)
    f(integral_constant<int, 6>{}, integral_constant<int, kColWide>{}, integral_constant<int, 2>{});
  else
    f(integral_constant<int, 8>{}, integral_constant<int, kColWide>{}, integral_constant<int, 2>{});
}

// Launch of one column-solve form: chunk depth en.col_kc,
// predictor or corrector, compute type T of the stencil inputs, arithmetic RA,
// flat ground or terrain.
template <class T, class RA, bool kTerr>
void launch_col_form(const Engine& en, int corrector, const ColArgs<T>& a, const char* name, cudaStream_t s) {
  const int nc = en.g64.nc;
  with_col_form(en.col_kc[corrector ? 1 : 0], en.col_narrow, [&](auto kc, auto cw, auto rl) {
    constexpr int KC = decltype(kc)::value, CW = decltype(cw)::value, RL = decltype(rl)::value;
    const unsigned blocks = (unsigned)((nc + CW - 1) / CW);
    if (corrector) {
      using F = ColForm<T, KC, CW, RL, true, kTerr>;
      ICON_CHAIN_SMEM(name, blocks, F::NT, F::bytes, s, (sn_column<T, RA, KC, CW, RL, 1, kTerr, false>), nc, en.v,
                       en.sc, 1, a);
    } else {
      using F = ColForm<T, KC, CW, RL, false, kTerr>;
      ICON_CHAIN_SMEM(name, blocks, F::NT, F::bytes, s, (sn_column<T, RA, KC, CW, RL, 0, kTerr, false>), nc, en.v,
                       en.sc, 0, a);
    }
  });
}

// The dynamic shared-memory limit of the forms of one (T, RA, kTerr).
template <class T, class RA, bool kTerr>
cudaError_t init_col_forms() {
  cudaError_t e = cudaSuccess;
  auto set = [&](auto kernel, size_t bytes) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  };
  // At most 196 of the 228 KB an SM as shared memory: the copies into the tiles
  // pass through L1, a line each for a chunk's 32 to 64 bytes of a row, and the
  // 28 KB that 228 leave hold too few lines in flight (mixed, R2B6 L90, the
  // predictor in chunks of 8: 2.18 ms with 228 KB, 1.59 with 196).
  auto carve = [&](auto kernel, size_t bytes, int blocks) {
    if (e == cudaSuccess && blocks * (bytes + 1024) > 164 * 1024)
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 85);
  };
  for (int kc : {0, 4, 6, 8})
    with_col_form(kc, kc == 0, [&](auto k, auto cw, auto rl) {
      constexpr int KC = decltype(k)::value, CW = decltype(cw)::value, RL = decltype(rl)::value;
      using P = ColForm<T, KC, CW, RL, false, kTerr>;
      using C = ColForm<T, KC, CW, RL, true, kTerr>;
      set(sn_column<T, RA, KC, CW, RL, 0, kTerr, false>, P::bytes);
      set(sn_column<T, RA, KC, CW, RL, 1, kTerr, false>, C::bytes);
      carve(sn_column<T, RA, KC, CW, RL, 0, kTerr, false>, P::bytes, P::blocks);
      carve(sn_column<T, RA, KC, CW, RL, 1, kTerr, false>, C::bytes, C::blocks);
    });
  return e;
}

// Kernel name of a launch (the profile tables and the autotuner key on it).
inline const char* column_name(bool mixed, bool f64col, bool terrain, int corrector) {
  if (!mixed) {
    if (terrain) return corrector ? "sn_column_corr_terrain" : "sn_column_pred_terrain";
    return corrector ? "sn_column_corr" : "sn_column_pred";
  }
  if (f64col) {
    if (terrain) return corrector ? "sn_column_corr_terrain_mx64" : "sn_column_pred_terrain_mx64";
    return corrector ? "sn_column_corr_mx64" : "sn_column_pred_mx64";
  }
  if (terrain) return corrector ? "sn_column_corr_terrain_mx" : "sn_column_pred_terrain_mx";
  return corrector ? "sn_column_corr_mx" : "sn_column_pred_mx";
}

}  // namespace
}  // namespace icon
