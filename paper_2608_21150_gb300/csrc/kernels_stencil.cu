// Stencil kernels of one dycore step (rows A1-A6, A8-A10).  The FP64 kernels
// stand here, with the edge kernels of the mixed modes that work a level at a
// time (row A12); the other FP32 kernels, four levels per thread, are in
// stencil_quad.cuh.
//
// Layout: level-contiguous X[h * ld + k] (k = 0 at the model top).  FP64: one
// thread per (horizontal point, level), flattened so that the 32 lanes of a
// warp cover consecutive levels of one or two columns.  Neighbour gathers
// X[nbr * ld + k] are coalesced runs of consecutive levels.
//
// Mixed mode: the stencils read FP32 mirrors of the state (vn, w and the
// perturbations rho - rho_ref, theta_v - theta_ref) and compute in FP32,
// except the exner difference of the horizontal pressure gradient (double-
// word); prognostic updates stay FP64 (the FP64 state plus an FP32 increment)
// and rewrite the mirrors; flux divergences are summed in double-word FP32 so
// that every edge flux is one value shared by its two cells (mass conserved
// to about 2^-48), and stored as the pair for the column solve.  FP64<->FP32
// conversions run on the FP64 pipe on this GPU, so they are done with integer
// operations, once per value by its writer, never per gather.
#include <cuda_runtime.h>

#include <initializer_list>
#include <type_traits>

#include "dfloat.cuh"
#include "fp64.cuh"
#include "kernels.h"

namespace icon {

thread_local Prof* g_prof = nullptr;

namespace {

template <class T>
constexpr bool kMixed = std::is_same<T, float>::value;

// FP64 <-> FP32 without the FP64 pipe (mixed mode): exact widening, and
// narrowing through the double-word split (round to nearest up to rare
// double-rounding ties)
__device__ __forceinline__ double f2d(float x) { return f2d_exact(x); }
__device__ __forceinline__ float d2f(double x) { return to_float(to_df(x)); }

__device__ __forceinline__ bool flat_index(int n_h, int nk, int& h, int& k) {
  const unsigned i = blockIdx.x * blockDim.x + threadIdx.x, q = i / (unsigned)nk;
  k = (int)(i - q * (unsigned)nk);
  h = (int)after_previous(q);
  return i < (unsigned)n_h * (unsigned)nk;
}

inline unsigned blocks_for(long long n, int threads) { return (unsigned)((n + threads - 1) / threads); }

// a * b + c with one rounding, in the compute type
__device__ __forceinline__ double fmat(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float fmat(float a, float b, float c) { return fmaf(a, b, c); }

// Second launch shape of va_edge_pre, va_cell_w, sn_cell_div and sn_edge_corr:
// one warp per horizontal point, its lanes striding over the levels, so the
// point's neighbour indices and weights are loaded once per warp.  The default
// of the FP32 sn_edge_corr; not of the FP64 kernels, where 90 levels fill only
// 90 of 96 lane slots of the saturated FP64 pipe (the tuner tries both).
__device__ __forceinline__ int warp_point() {
  return (int)after_previous(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
}
__device__ __forceinline__ int lane_id() { return (int)(threadIdx.x & 31u); }
inline unsigned blocks_for_points(long long n_points, int threads) {
  const int warps = threads / 32;
  return (unsigned)((n_points + warps - 1) / warps);
}
// CTAs of a two-shape kernel: shape 1 one warp per point, 0 one thread per (point, level)
inline unsigned blocks_by_shape(int shape, long long n_h, int nk, int threads) {
  return shape ? blocks_for_points(n_h, threads) : blocks_for(n_h * nk, threads);
}

constexpr int kThreads = 256;

// threads per CTA of stencil kernel `id` from the autotuner's table (0: default)
inline int tuned(const int* threads, int id) { return threads && threads[id] > 0 ? threads[id] : kThreads; }
#define TH(id) tuned(threads, id)
// tile shape of a two-shape kernel from the autotuner's table (-1: the
// compute type's default, one warp per point in FP32, one thread per
// (point, level) in FP64)
template <class T>
inline int shaped(const int* shapes, int id) {
  return shapes && shapes[id] >= 0 ? shapes[id] : (kMixed<T> ? 1 : 0);
}
#define SH(id) shaped<T>(shapes, id)

template <class T>
const char* kname(const char* f64, const char* f32) {
  return kMixed<T> ? f32 : f64;
}

}  // namespace
}  // namespace icon
#include "stencil_quad.cuh"
namespace icon {
namespace {

// -------------------------------------------------------------------------
// A1: tangential wind and edge kinetic energy
//   vt = sum_j vt_w[j] vn[e_j] (Perot reconstruction averaged over the two
//   cells, projected on t_e), K_e = (vn^2 + vt^2)/2, stored as 2 K_e (the
//   1/2 is folded into the gradient's stored factor 1/(2 d_e))
// -------------------------------------------------------------------------
// Also vn at the half levels, vn_ie (interpolated inside with the level
// weights -- the edge weights wgt_e over terrain -- the top level's value at the
// top and the lowest level's at the ground), for the edge tendency kernel.
// Both tile shapes evaluate every (edge, level) with the same explicit FMAs
// (va_edge_pre_at), so the autotuner's choice of shape does not change a bit.
__device__ __forceinline__ void va_edge_pre_at(const VertT<double>& v, int e, int k, int nlev, const double* x0,
                                               const double* x1, const double* x2, const double* x3, const double* x4,
                                               const double* w, double* vt, double* ekin, double* vn_ie,
                                               const double* wgt_e) {
  const int nlevp = nlev + 1;
  const double vne = x0[k];
  double t = w[0] * vne;
  t = fmat(w[1], x1[k], t);
  t = fmat(w[2], x2[k], t);
  t = fmat(w[3], x3[k], t);
  t = fmat(w[4], x4[k], t);
  vt[(size_t)e * nlev + k] = t;
  ekin[(size_t)e * nlev + k] = fmat(vne, vne, t * t);
  const double wg = wgt_e ? wgt_e[(size_t)e * nlevp + k] : v.wgt[k];
  vn_ie[(size_t)e * nlevp + k] = k == 0 ? vne : fmat(wg, x0[k - 1] - vne, vne);
  if (k == nlev - 1) vn_ie[(size_t)e * nlevp + nlev] = vne;
}

__global__ void va_edge_pre(GridT<double> g, VertT<double> v, const double* __restrict__ vn, double* __restrict__ vt,
                            double* __restrict__ ekin, double* __restrict__ vn_ie, const double* __restrict__ wgt_e,
                            int shape) {
  const int nlev = v.nlev;
  if (shape) {  // one warp per edge, its lanes over the levels
    const int e = warp_point();
    if (e >= g.ne) return;
    const double* w = g.vt_w + 5 * (size_t)e;
    const double wl[5] = {w[0], w[1], w[2], w[3], w[4]};
    const int* q = g.e2c2e + 4 * (size_t)e;
    const double* x0 = vn + (size_t)e * nlev;
    const double* x1 = vn + (size_t)q[0] * nlev;
    const double* x2 = vn + (size_t)q[1] * nlev;
    const double* x3 = vn + (size_t)q[2] * nlev;
    const double* x4 = vn + (size_t)q[3] * nlev;
    for (int k = lane_id(); k < nlev; k += 32) va_edge_pre_at(v, e, k, nlev, x0, x1, x2, x3, x4, wl, vt, ekin, vn_ie, wgt_e);
    return;
  }
  int e, k;
  if (!flat_index(g.ne, nlev, e, k)) return;
  const int* q = g.e2c2e + 4 * (size_t)e;
  va_edge_pre_at(v, e, k, nlev, vn + (size_t)e * nlev, vn + (size_t)q[0] * nlev, vn + (size_t)q[1] * nlev,
                 vn + (size_t)q[2] * nlev, vn + (size_t)q[3] * nlev, g.vt_w + 5 * (size_t)e, vt, ekin, vn_ie, wgt_e);
}

// -------------------------------------------------------------------------
// A1-A2 over terrain: contravariant correction at cell half levels, the
// vertical velocity of a parcel that follows the coordinate surface,
//   wcc = sum_e q_e (vn_ie dz/dn + vt_ie dz/dt)
// with vn, vt interpolated to the edge half levels by the edge weights (the
// lowest full level's values at the ground; vn_ie from va_edge_pre; the
// slopes vanish at the flat model top, where wcc = 0).
// -------------------------------------------------------------------------
__global__ void va_concorr(GridT<double> g, VertT<double> v, TerrT<double> tr, const double* __restrict__ vn_ie,
                           const double* __restrict__ vt, double* __restrict__ wcc) {
  int c, k;
  const int nlev = v.nlev, nlevp = nlev + 1;
  if (!flat_index(g.nc, nlevp, c, k)) return;
  double s = 0;
  if (k > 0) {
    const int* ce = g.c2e + 3 * (size_t)c;
    const double* q = g.e2c_w + 3 * (size_t)c;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int e = ce[j];
      const double* y = vt + (size_t)e * nlev;
      const size_t ih = (size_t)e * nlevp + k;
      const double a = vn_ie[ih];
      const double b = k == nlev ? y[nlev - 1] : y[k] + tr.wgt_e[ih] * (y[k - 1] - y[k]);
      s += q[j] * (a * tr.ddxn_ifc[ih] + b * tr.ddxt_ifc[ih]);
    }
  }
  wcc[(size_t)c * nlevp + k] = s;
}

// -------------------------------------------------------------------------
// A2: cells: K_c = sum q_e K_e  (and, in the corrector, the divergence-damping
//     Laplacian dd2 = lapc(div vn*));  vertices: zeta = curl vn (full levels),
//     w_v = sum r_c w_c (half levels).  One launch over nc*nlev + nv*(nlev+1).
// -------------------------------------------------------------------------
// Also, per cell and full level, wq = w_k + w_k+1 (over terrain the
// contravariant w - wcc): the edge tendency's mean of four w is then the
// sum of its two cells' wq, computed once per cell instead of once per edge.
// In FP64 the Laplacian is sum L_j dd_j - (sum L_j) dd_c: fewer FP64
// operations (the damping increment is a small part of vn, so the
// cancellation in the sum costs nothing measurable); FP32 keeps the
// differences.
__global__ void va_cell_vert(GridT<double> g, VertT<double> v, const double* __restrict__ vn,
                             const double* __restrict__ w, const double* __restrict__ ekin_e,
                             double* __restrict__ ekin_c, const double* __restrict__ divd, double* __restrict__ divd2,
                             double* __restrict__ zeta, double* __restrict__ w_v, double* __restrict__ wq,
                             const double* __restrict__ wcc) {
  const int nlev = v.nlev, nlevp = nlev + 1;
  unsigned i = flat_thread();
  const unsigned ncell = (unsigned)g.nc * nlev;
  if (i < ncell) {
    int c = (int)(i / (unsigned)nlev), k = (int)(i - (unsigned)c * nlev);
    const int* ce = g.c2e + 3 * (size_t)c;
    const double* q = g.e2c_w + 3 * (size_t)c;
    double s = q[0] * ekin_e[(size_t)ce[0] * nlev + k];
    s += q[1] * ekin_e[(size_t)ce[1] * nlev + k];
    s += q[2] * ekin_e[(size_t)ce[2] * nlev + k];
    ekin_c[i] = s;
    const double* wc = w + (size_t)c * nlevp;
    if (wcc) {
      const double* qc = wcc + (size_t)c * nlevp;
      wq[i] = (wc[k] - qc[k]) + (wc[k + 1] - qc[k + 1]);
    } else {
      wq[i] = wc[k] + wc[k + 1];
    }
    if (divd2) {
      const int* cc = g.c2e2c + 3 * (size_t)c;
      const double* L = g.lap_c + 3 * (size_t)c;
      const double dc = divd[i];
      const double d0 = divd[(size_t)cc[0] * nlev + k], d1 = divd[(size_t)cc[1] * nlev + k],
              d2 = divd[(size_t)cc[2] * nlev + k];
      divd2[i] = fmat(L[2], d2, fmat(L[1], d1, fmat(L[0], d0, -(g.lap_s[c] * dc))));
    }
    return;
  }
  i -= ncell;
  if (i >= (unsigned)g.nv * nlevp) return;
  int vx = (int)(i / (unsigned)nlevp), k = (int)(i - (unsigned)vx * nlevp);
  const int* ve = g.v2e + 6 * (size_t)vx;
  const int* vc = g.v2c + 6 * (size_t)vx;
  const double* cw = g.curl_v + 6 * (size_t)vx;
  const double* rw = g.c2v_w + 6 * (size_t)vx;
  if (k < nlev) {
    double z = 0;
#pragma unroll
    for (int j = 0; j < 6; ++j) z += cw[j] * vn[(size_t)ve[j] * nlev + k];
    zeta[(size_t)vx * nlev + k] = z;
  }
  double s = 0;
#pragma unroll
  for (int j = 0; j < 6; ++j) s += rw[j] * w[(size_t)vc[j] * nlevp + k];
  w_v[i] = s;
}

// -------------------------------------------------------------------------
// A3: vn advective tendency (full levels) and horizontal advection of w at
//     edges (interior half levels); one launch over ne*(nlev+1).
//   ddt_vn = -(K_c1 - K_c0)/d + (zeta_e + f) vt - wbar (vn_ie_k - vn_ie_k+1)/dz
//   gw_e   = vn_ie (w_c1 - w_c0)/d + vt_ie (w_vp - w_vm)/l
// -------------------------------------------------------------------------
// Over terrain (kTerr): edge interpolation weights and layer thicknesses, and
// the contravariant velocity w - wcc as the advecting vertical velocity.
// Arithmetic arranged for few FP64 instructions (the FP64 mode is bound by
// GB300's FP64 issue rate): wbar dvn/dz = (wq_c0 + wq_c1) (vn_ie_k -
// vn_ie_k+1) dz^-1/4 with the cells' sums of two w from va_cell_vert and
// dz^-1/4 stored, the Coriolis term's 1/2 folded into a multiply-add, the
// gradient of 2K times 1/(2 d) into the final multiply-add.  gw_e is stored
// times d_e (its 1/d_e is folded into va_cell_w's weights).
template <bool kTerr = false>
__global__ void va_edge_tend(GridT<double> g, VertT<double> v, const double* __restrict__ vn_ie,
                             const double* __restrict__ w, const double* __restrict__ vt,
                             const double* __restrict__ ekin_c, const double* __restrict__ zeta,
                             const double* __restrict__ w_v, double* __restrict__ ddt_vn, double* __restrict__ gw_e,
                             TerrT<double> tr, const double* __restrict__ wq) {
  int e, k;
  const int nlev = v.nlev, nlevp = nlev + 1;
  if (!flat_index(g.ne, nlevp, e, k)) return;
  const int c0 = g.e2c[2 * e], c1 = g.e2c[2 * e + 1];
  const double* vte = vt + (size_t)e * nlev;
  const double vnie_k = vn_ie[(size_t)e * nlevp + k];
  if (k < nlev) {
    const int vm = g.e2v[2 * e], vp = g.e2v[2 * e + 1];
    const double vnie_k1 = vn_ie[(size_t)e * nlevp + k + 1];
    const double ws = wq[(size_t)c0 * nlev + k] + wq[(size_t)c1 * nlev + k];
    const double qdz = kTerr ? tr.qdz_e[(size_t)e * nlev + k] : v.qdz[k];
    const double adv = (ws * (vnie_k - vnie_k1)) * qdz;
    const double zf = fmat(double(0.5), zeta[(size_t)vm * nlev + k] + zeta[(size_t)vp * nlev + k], g.f_e[e]);
    const double dk = ekin_c[(size_t)c0 * nlev + k] - ekin_c[(size_t)c1 * nlev + k];
    ddt_vn[(size_t)e * nlev + k] = fmat(dk, g.hinv_d[e], fmat(zf, vte[k], -adv));
  }
  double gw = 0;
  if (k > 0 && k < nlev) {
    const int vm = g.e2v[2 * e], vp = g.e2v[2 * e + 1];
    const double wg = kTerr ? tr.wgt_e[(size_t)e * nlevp + k] : v.wgt[k];
    const double vtie = vte[k] + wg * (vte[k - 1] - vte[k]);
    const double dwn = w[(size_t)c1 * nlevp + k] - w[(size_t)c0 * nlevp + k];
    const double dwt = (w_v[(size_t)vp * nlevp + k] - w_v[(size_t)vm * nlevp + k]) * g.d_o_l[e];
    gw = fmat(vnie_k, dwn, vtie * dwt);
  }
  gw_e[(size_t)e * nlevp + k] = gw;
}

// -------------------------------------------------------------------------
// A4: w advective tendency at interior half levels (0 at top and ground)
//   ddt_w = -sum q_e gw_e - w (wf_{k-1} - wf_k)/dzh,  wf full-level averages
//   (q_e/d_e stored: gw_e holds the advection times d_e)
// -------------------------------------------------------------------------
// Over terrain (kTerr): advected by w - wcc, per-cell half-level spacing.
// Both tile shapes evaluate every (cell, half level) with va_cell_w_at.
template <bool kTerr>
__device__ __forceinline__ double va_cell_w_at(const VertT<double>& v, const TerrT<double>& tr, int c, int k, int nlev,
                                               const double* g0, const double* g1, const double* g2, const double* q,
                                               const double* wc, const double* wcc) {
  if (k == 0 || k >= nlev) return double(0);
  const double h = fmat(q[2], g2[k], fmat(q[1], g1[k], q[0] * g0[k]));
  // the difference of the full-level means above and below, (w_k-1 - w_k+1) / 2,
  // with the 1/2 folded into the stored 1/(2 dzh)
  double wa, qd;
  if constexpr (kTerr) {
    const size_t ih = (size_t)c * (nlev + 1) + k;
    wa = wc[k] - wcc[ih];
    qd = tr.qdzh_c[ih];
  } else {
    wa = wc[k];
    qd = v.qdzh[k];
  }
  return fmat(-(wa * (wc[k - 1] - wc[k + 1])), qd, -h);
}

template <bool kTerr = false>
__global__ void va_cell_w(GridT<double> g, VertT<double> v, const double* __restrict__ w,
                          const double* __restrict__ gw_e, double* __restrict__ ddt_w, TerrT<double> tr,
                          const double* __restrict__ wcc, int shape) {
  const int nlev = v.nlev, nlevp = nlev + 1;
  if (shape) {  // one warp per cell, its lanes over the half levels
    const int c = warp_point();
    if (c >= g.nc) return;
    const int* ce = g.c2e + 3 * (size_t)c;
    const double* qp = g.e2c_wd + 3 * (size_t)c;
    const double q[3] = {qp[0], qp[1], qp[2]};
    const double* g0 = gw_e + (size_t)ce[0] * nlevp;
    const double* g1 = gw_e + (size_t)ce[1] * nlevp;
    const double* g2 = gw_e + (size_t)ce[2] * nlevp;
    const double* wc = w + (size_t)c * nlevp;
    for (int k = lane_id(); k < nlevp; k += 32)
      ddt_w[(size_t)c * nlevp + k] = va_cell_w_at<kTerr>(v, tr, c, k, nlev, g0, g1, g2, q, wc, wcc);
    return;
  }
  int c, k;
  if (!flat_index(g.nc, nlevp, c, k)) return;
  const int* ce = g.c2e + 3 * (size_t)c;
  ddt_w[(size_t)c * nlevp + k] =
      va_cell_w_at<kTerr>(v, tr, c, k, nlev, gw_e + (size_t)ce[0] * nlevp, gw_e + (size_t)ce[1] * nlevp,
                             gw_e + (size_t)ce[2] * nlevp, g.e2c_wd + 3 * (size_t)c, w + (size_t)c * nlevp, wcc);
}

// -------------------------------------------------------------------------
// A1-A4 in one launch (mixed precision, flat ground): one CTA per patch of
// consecutive cells (the refinement order makes patches compact), chunks of
// kVaL levels.  Per chunk, vn on every edge the patch reads and w on every
// cell it reads come into shared memory (coalesced runs of levels); then, one
// thread per edge, cell or vertex looping over the chunk's levels: vt and 2K
// on the edges of the patch's cells and their neighbours, 2K at those cells,
// vorticity and w at the vertices, the vn tendency and w's horizontal
// advection on the own cells' edges, the w tendency of the own cells -- each
// stage from shared memory, where the four kernels above pass through HBM.
// Results are staged in shared memory and stored as runs of levels.  Halo
// values are computed again by every patch that needs them; an edge's
// tendency and vt are written by the patch of its first cell.  Local indices
// and the grid factors come in patch order (16-bit index rows, FP32 factor
// rows), so every item's table is one or two vector loads per chunk.  Every
// value is the same expression as in the four kernels (the same bits).
// -------------------------------------------------------------------------
constexpr int kVaL = 8;          // levels per chunk
constexpr int kVaS = kVaL + 1;   // shared-memory stride of a per-item run of L or L + 1 levels (odd)
constexpr int kVaSn = kVaL + 3;  // stride of the staged vn and w runs of L + 2 levels (odd)
constexpr int kVaThreads = 512;

__host__ __device__ inline size_t va_fused_smem_floats(int max_e0, int max_e1, int max_c3, int max_c0, int max_v3,
                                                       int max_e4) {
  return 2 * (size_t)kVaSn * ((size_t)max_e0 + max_c0) +
         (size_t)kVaS * (2 * (size_t)max_e1 + 2 * (size_t)max_e4 + max_c3 + 2 * (size_t)max_v3);
}

__device__ __forceinline__ int lo16(unsigned x) { return (int)(x & 0xffffu); }
__device__ __forceinline__ int hi16(unsigned x) { return (int)(x >> 16); }

// 4-byte asynchronous global->shared copy; cp_commit closes the thread's
// group, cp_wait_all waits for every group it issued
__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

__global__ void __launch_bounds__(kVaThreads, 2) va_fused(GridT<float> g, VertT<float> v, VaPatchT pt,
                                                          const float* __restrict__ vn, const float* __restrict__ w,
                                                          float* __restrict__ vt_out, float* __restrict__ ddt_vn,
                                                          float* __restrict__ ddt_w, const float* __restrict__ divd,
                                                          float* __restrict__ divd2) {
  extern __shared__ float sf[];
  constexpr int L = kVaL, S = kVaS, Sn = kVaSn;
  const int p = (int)after_previous(blockIdx.x);
  const int nlev = v.nlev, ld = v.ldf;
  const int e0a = pt.off_e0[p], ne0 = pt.off_e0[p + 1] - e0a;
  const int e1a = pt.off_e1[p], ne1 = pt.off_e1[p + 1] - e1a;
  const int c0a = pt.off_c0[p], nc0 = pt.off_c0[p + 1] - c0a, nc3 = pt.n_c3[p];
  const int v3a = pt.off_v3[p], nv3 = pt.off_v3[p + 1] - v3a;
  const int e4a = pt.off_e4[p], ne4 = pt.off_e4[p + 1] - e4a, nw4 = pt.n_w4[p];
  const int c_begin = p * pt.P, ncown = min(pt.P, g.nc - c_begin);
  // two stages of [e0][Sn] vn at full levels k0-1 .. k0+L and [c0][Sn] w at
  // half levels k0-1 .. k0+L: the next chunk's copies run during this one
  const size_t stage = (size_t)(pt.max_e0 + pt.max_c0) * Sn;
  float* vt_s = sf + 2 * stage;                // [e1][S]: vt at full levels k0-1 .. k0+L-1
  float* ek_s = vt_s + (size_t)pt.max_e1 * S;  // [e1][S]: 2K at full levels k0 .. k0+L-1; then ddt_vn of E4
  float* vi_s = ek_s + (size_t)pt.max_e1 * S;  // [e4][S]: vn at half levels k0 .. k0+L
  float* gw_s = vi_s + (size_t)pt.max_e4 * S;  // [e4][S]: w's horizontal advection, half levels k0 .. k0+L-1
  float* kc_s = gw_s + (size_t)pt.max_e4 * S;  // [c3][S]: 2K at the cells; then ddt_w of the own cells
  float* ze_s = kc_s + (size_t)pt.max_c3 * S;  // [v3][S]: vorticity, full levels
  float* wv_s = ze_s + (size_t)pt.max_v3 * S;  // [v3][S]: w at the vertices, half levels
  float* dv_s = ek_s;
  float* dw_s = kc_s;
  // consecutive threads copy consecutive levels of one row (coalesced)
  auto issue = [&](int kc, float* vs) {
    float* ws = vs + (size_t)pt.max_e0 * Sn;
    for (int i = threadIdx.x; i < (ne0 + nc0) * (L + 2); i += blockDim.x) {
      const int it = i / (L + 2), lv = i - it * (L + 2);
      if (it < ne0) {
        const int k = min(max(kc - 1 + lv, 0), nlev - 1);
        cp_async4(vs + it * Sn + lv, vn + (size_t)pt.e0_g[e0a + it] * ld + k);
      } else {
        const int kh = min(max(kc - 1 + lv, 0), nlev);
        const int ic = it - ne0;
        cp_async4(ws + ic * Sn + lv, w + (size_t)pt.c0_g[c0a + ic] * ld + kh);
      }
    }
    cp_commit();
  };
  issue(0, sf);
  for (int k0 = 0, b = 0; k0 <= nlev + L; k0 += L, b ^= 1) {
    cp_wait_all();
    __syncthreads();
    if (k0 > 0) {  // the previous chunk's w tendencies (own cells), coalesced along the levels
      const int kp = k0 - L;
      for (int i = threadIdx.x; i < ncown * L; i += blockDim.x) {
        const int it = i / L, lv = i - it * L, k = kp + lv;
        if (k <= nlev) ddt_w[(size_t)(c_begin + it) * ld + k] = dw_s[it * S + lv];
      }
    }
    if (k0 > nlev) break;
    if (k0 + L <= nlev) issue(k0 + L, sf + (b ^ 1) * stage);
    const float* vn_s = sf + b * stage;
    const float* w_s = vn_s + (size_t)pt.max_e0 * Sn;
    // A1: vt and 2K on the E1 edges; vn at the half levels of the E4 edges
    for (int i = threadIdx.x; i < ne1 + ne4; i += blockDim.x) {
      if (i < ne1) {
        const int it = i;
        const uint4 nb = *reinterpret_cast<const uint4*>(pt.e1_i + 8 * (size_t)(e1a + it));
        const float* n0 = vn_s + lo16(nb.x) * Sn;
        const float* n1 = vn_s + hi16(nb.x) * Sn;
        const float* n2 = vn_s + lo16(nb.y) * Sn;
        const float* n3 = vn_s + hi16(nb.y) * Sn;
        const float* n4 = vn_s + lo16(nb.z) * Sn;
        const float* wt = pt.e1_w + 5 * (size_t)(e1a + it);
        const float w0 = wt[0], w1 = wt[1], w2 = wt[2], w3 = wt[3], w4 = wt[4];
#pragma unroll
        for (int lv = 0; lv <= L; ++lv) {
          const int k = k0 - 1 + lv;
          if (k < 0 || k >= nlev) continue;
          const float vne = n0[lv];
          float t = w0 * vne;
          t = fmat(w1, n1[lv], t);
          t = fmat(w2, n2[lv], t);
          t = fmat(w3, n3[lv], t);
          t = fmat(w4, n4[lv], t);
          vt_s[it * S + lv] = t;
          if (lv >= 1) ek_s[it * S + lv - 1] = fmat(vne, vne, t * t);
        }
      } else {
        const int it = i - ne1;
        const float* x = vn_s + (int)pt.e4_i[8 * (size_t)(e4a + it) + 1] * Sn;
#pragma unroll
        for (int lv = 0; lv <= L; ++lv) {
          const int kh = k0 + lv;
          if (kh > nlev) break;
          float vi;
          if (kh == 0) {
            vi = x[lv + 1];
          } else if (kh == nlev) {
            vi = x[lv];
          } else {
            const float vne = x[lv + 1];
            vi = fmat(v.wgt[kh], x[lv] - vne, vne);
          }
          vi_s[it * S + lv] = vi;
        }
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nw4 * L; i += blockDim.x) {  // vt of the edges this patch writes
      const int it = i / L, lv = i - it * L, k = k0 + lv;
      if (k < nlev) vt_out[(size_t)pt.e4_g[e4a + it] * ld + k] = vt_s[(int)pt.e4_i[8 * (size_t)(e4a + it)] * S + lv + 1];
    }
    if (divd2) {  // the corrector's divergence-damping Laplacian at the own cells
      for (int i = threadIdx.x; i < ncown * L; i += blockDim.x) {
        const int it = i / L, lv = i - it * L, k = k0 + lv;
        if (k >= nlev) continue;
        const int c = c_begin + it;
        const int* cc = g.c2e2c + 3 * (size_t)c;
        const float* Lw = g.lap_c + 3 * (size_t)c;
        const size_t ic = (size_t)c * ld + k;
        const float dc = divd[ic];
        const float d0 = divd[(size_t)cc[0] * ld + k], d1 = divd[(size_t)cc[1] * ld + k],
                    d2 = divd[(size_t)cc[2] * ld + k];
        float r = Lw[0] * (d0 - dc);
        r += Lw[1] * (d1 - dc);
        r += Lw[2] * (d2 - dc);
        divd2[ic] = r;
      }
    }
    // A2: 2K at the C3 cells (all levels of the chunk); vorticity and w at the
    // V3 vertices (each vertex in two halves of the chunk's levels)
    for (int i = threadIdx.x; i < nc3 + 2 * nv3; i += blockDim.x) {
      if (i < nc3) {
        const int it = i;
        const uint2 ce = *reinterpret_cast<const uint2*>(pt.c3_i + 4 * (size_t)(c0a + it));
        const float* k0p = ek_s + lo16(ce.x) * S;
        const float* k1p = ek_s + hi16(ce.x) * S;
        const float* k2p = ek_s + lo16(ce.y) * S;
        const float4 q = *reinterpret_cast<const float4*>(pt.c3_w + 4 * (size_t)(c0a + it));
#pragma unroll
        for (int lv = 0; lv < L; ++lv) {
          const int k = k0 + lv;
          if (k >= nlev) break;
          float sk = q.x * k0p[lv];
          sk += q.y * k1p[lv];
          sk += q.z * k2p[lv];
          kc_s[it * S + lv] = sk;
        }
      } else {
        const int it = (i - nc3) >> 1, l0 = ((i - nc3) & 1) * (L / 2);
        const uint4* xi = reinterpret_cast<const uint4*>(pt.v3_i + 16 * (size_t)(v3a + it));
        const uint4 xa = xi[0], xb = xi[1];
        const float4* wp = reinterpret_cast<const float4*>(pt.v3_w + 12 * (size_t)(v3a + it));
        const float4 wa = wp[0], wb = wp[1], wc = wp[2];
        const float* ep[6] = {vn_s + lo16(xa.x) * Sn + 1, vn_s + hi16(xa.x) * Sn + 1, vn_s + lo16(xa.y) * Sn + 1,
                              vn_s + hi16(xa.y) * Sn + 1, vn_s + lo16(xa.z) * Sn + 1, vn_s + hi16(xa.z) * Sn + 1};
        const float* cp[6] = {w_s + lo16(xa.w) * Sn + 1, w_s + hi16(xa.w) * Sn + 1, w_s + lo16(xb.x) * Sn + 1,
                              w_s + hi16(xb.x) * Sn + 1, w_s + lo16(xb.y) * Sn + 1, w_s + hi16(xb.y) * Sn + 1};
        const float cwl[6] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y};
        const float rwl[6] = {wb.z, wb.w, wc.x, wc.y, wc.z, wc.w};
#pragma unroll
        for (int j = 0; j < L / 2; ++j) {
          const int lv = l0 + j, k = k0 + lv;
          if (k > nlev) break;
          if (k < nlev) {
            float z = 0;
#pragma unroll
            for (int m = 0; m < 6; ++m) z += cwl[m] * ep[m][lv];
            ze_s[it * S + lv] = z;
          }
          float sw = 0;
#pragma unroll
          for (int m = 0; m < 6; ++m) sw += rwl[m] * cp[m][lv];
          wv_s[it * S + lv] = sw;
        }
      }
    }
    __syncthreads();
    // A3: the vn tendency (edges this patch writes) and w's horizontal
    // advection (times d) on the E4 edges, each edge in two halves of the levels
    for (int i = threadIdx.x; i < 2 * ne4; i += blockDim.x) {
      const int it = i >> 1, l0 = (i & 1) * (L / 2);
      const uint4 x = *reinterpret_cast<const uint4*>(pt.e4_i + 8 * (size_t)(e4a + it));
      const float4 cf = *reinterpret_cast<const float4*>(pt.e4_w + 4 * (size_t)(e4a + it));
      const float* vt1 = vt_s + lo16(x.x) * S;
      const int lc0 = lo16(x.y), lc1 = hi16(x.y);
      const float* kc0 = kc_s + lc0 * S;
      const float* kc1 = kc_s + lc1 * S;
      const float* w0 = w_s + lc0 * Sn;
      const float* w1 = w_s + lc1 * Sn;
      const float* zm = ze_s + lo16(x.z) * S;
      const float* zp = ze_s + hi16(x.z) * S;
      const float* wvm = wv_s + lo16(x.z) * S;
      const float* wvp = wv_s + hi16(x.z) * S;
      const bool own = it < nw4;
      const float* vie = vi_s + it * S;
#pragma unroll
      for (int j = 0; j < L / 2; ++j) {
        const int lv = l0 + j, k = k0 + lv;
        if (k > nlev) break;
        const float vnie_k = vie[lv];
        if (k < nlev && own) {
          const float vnie_k1 = vie[lv + 1];
          const float ws = (w0[lv + 1] + w0[lv + 2]) + (w1[lv + 1] + w1[lv + 2]);
          const float adv = (ws * (vnie_k - vnie_k1)) * v.qdz[k];
          const float zf = fmat(0.5f, zm[lv] + zp[lv], cf.x);
          const float dk = kc0[lv] - kc1[lv];
          dv_s[it * S + lv] = fmat(dk, cf.y, fmat(zf, vt1[lv + 1], -adv));
        }
        float gw = 0;
        if (k > 0 && k < nlev) {
          const float wg = v.wgt[k];
          const float vtk = vt1[lv + 1];
          const float vtie = vtk + wg * (vt1[lv] - vtk);
          const float dwn = w1[lv + 1] - w0[lv + 1];
          const float dwt = (wvp[lv] - wvm[lv]) * cf.z;
          gw = fmat(vnie_k, dwn, vtie * dwt);
        }
        gw_s[it * S + lv] = gw;
      }
    }
    __syncthreads();
    // A4: the w tendency of the own cells, each cell in four quarters of the
    // levels (stored at the next chunk's start); the vn tendencies of the
    // edges this patch writes
    for (int i = threadIdx.x; i < 4 * ncown; i += blockDim.x) {
      const int it = i >> 2, l0 = (i & 3) * (L / 4);
      const int c = c_begin + it;
      const uint2 ce = *reinterpret_cast<const uint2*>(pt.own_i + 4 * (size_t)c);
      const float* g0 = gw_s + lo16(ce.x) * S;
      const float* g1 = gw_s + hi16(ce.x) * S;
      const float* g2 = gw_s + lo16(ce.y) * S;
      const float4 q = *reinterpret_cast<const float4*>(pt.own_w + 4 * (size_t)c);
      const float* wc = w_s + it * Sn;  // wc[lv + 1]: half level k0 + lv
#pragma unroll
      for (int j = 0; j < L / 4; ++j) {
        const int lv = l0 + j, k = k0 + lv;
        if (k > nlev) break;
        float r = 0.0f;
        if (k > 0 && k < nlev) {
          const float h = fmat(q.z, g2[lv], fmat(q.y, g1[lv], q.x * g0[lv]));
          const float wa = wc[lv + 1];
          r = fmat(-(wa * (wc[lv] - wc[lv + 2])), v.qdzh[k], -h);
        }
        dw_s[it * S + lv] = r;
      }
    }
    for (int i = threadIdx.x; i < nw4 * L; i += blockDim.x) {
      const int it = i / L, lv = i - it * L, k = k0 + lv;
      if (k < nlev) ddt_vn[(size_t)pt.e4_g[e4a + it] * ld + k] = dv_s[it * S + lv];
    }
  }
}

// -------------------------------------------------------------------------
// A5 (predictor): Green-Gauss gradients of rho and theta_v as four planes
// grad4 [4][nc*nlev].  FP64: the coefficients (A, B) of both in the cell's own
// basis, grad = G_a A + G_b B with two of the three vectors of
// grad = sum_j G_j (psi_j - psi_c): with G_m = alpha G_a + beta G_b,
// A = psi_a + alpha psi_m - (1 + alpha) psi_c, two FP64 operations a component
// where the cell frame's x and y take four, and the edge kernel's offsets are
// stored in that basis too (upw_s).  The pair (a, b) is the least parallel one,
// so |alpha|, |beta| <= 1 and the sums cancel no more than the frame's did.
// 327680 cells of 90 levels: 1028 -> 619 us.  (Mixed mode: x and y of the
// perturbations, in stencil_quad.cuh.)
// -------------------------------------------------------------------------
// exner_ref_c: the per-column reference exner over terrain (kTerr).
template <bool kTerr = false>
__global__ void sn_cell_grad(GridT<double> g, VertT<double> v, const double* __restrict__ rho,
                             const double* __restrict__ theta, double* __restrict__ grad4,
                             const double* __restrict__ exner, const double* __restrict__ exner_pr, double exfac,
                             double* __restrict__ pex, const double* __restrict__ exner_ref_c) {
  int c, k;
  const int nlev = v.nlev;
  if (!flat_index(g.nc, nlev, c, k)) return;
  const size_t n = (size_t)g.nc * nlev;
  const int* cc = g.grad_nb + 3 * (size_t)c;
  const double* G = g.grad_b + 4 * (size_t)c;
  const size_t i = (size_t)c * nlev + k;
  const double ex_ref = kTerr ? exner_ref_c[i] : v.exner_ref[k];
  // extrapolated exner perturbation (1 + a) pr - a pr_old of this cell, for the
  // pressure gradient at its edges
  pex[i] = (1.0 + exfac) * (exner[i] - ex_ref) - exfac * exner_pr[i];
  const size_t ia = (size_t)cc[0] * nlev + k, ib = (size_t)cc[1] * nlev + k, im = (size_t)cc[2] * nlev + k;
  const double r = rho[i], rm = rho[im], t = theta[i], tm = theta[im];
  grad4[i] = fma(G[0], rm, fma(-G[2], r, rho[ia]));
  grad4[n + i] = fma(G[1], rm, fma(-G[3], r, rho[ib]));
  grad4[2 * n + i] = fma(G[0], tm, fma(-G[2], t, theta[ia]));
  grad4[3 * n + i] = fma(G[1], tm, fma(-G[3], t, theta[ib]));
}

// The same planes read back: from (A, B) to the x and y of the cell's frame, in
// place, each a sum of two rounded products.
__global__ void gradient_frame(GridT<double> g, int nlev, double* __restrict__ f) {
  int c, k;
  if (!flat_index(g.nc, nlev, c, k)) return;
  const size_t n = (size_t)g.nc * nlev;
  const int m = g.grad_m[c], a = (m + 1) % 3, b = (m + 2) % 3;
  const double* G = g.grad_c + 6 * (size_t)c;
  double* p = f + (size_t)c * nlev + k;
#pragma unroll
  for (int j = 0; j < 2; ++j, p += 2 * n) {
    const double ga = p[0], gb = p[n];
    p[0] = __dadd_rn(__dmul_rn(G[2 * a], ga), __dmul_rn(G[2 * b], gb));
    p[n] = __dadd_rn(__dmul_rn(G[2 * a + 1], ga), __dmul_rn(G[2 * b + 1], gb));
  }
}

// -------------------------------------------------------------------------
// A6 (predictor edges): upwind rho_e/theta_e from the back trajectory over
// dt/2, horizontal pressure gradient with the extrapolated exner perturbation,
// and the vn predictor, FP64 (the mixed modes: sn_edge_pred_q in
// stencil_quad.cuh).  The extrapolated exner perturbations come per cell from
// sn_cell_grad; their difference across the edge is taken in FP64, since
// neighbouring perturbations agree to 4-5 digits.
// -------------------------------------------------------------------------
// Over terrain (kTerr) the pressure gradient is taken along the true
// horizontal: the along-level difference minus the slope of the full level
// times the edge mean of the two cells' vertical derivatives (centred, one-
// sided at the top and the ground) of the extrapolated exner perturbation.
template <bool kTerr = false>
__global__ void sn_edge_pred(GridT<double> g, VertT<double> v, ScalT<double> sc, const double* __restrict__ vn,
                             const double* __restrict__ vt, const double* __restrict__ ddt_vn,
                             const double* __restrict__ rho, const double* __restrict__ theta,
                             const double* __restrict__ pex, const double* __restrict__ cid64,
                             const double* __restrict__ grad4, double* __restrict__ rho_e, double* __restrict__ theta_e,
                             double* __restrict__ hpg, double* __restrict__ vn_p, TerrT<double> tr) {
  int e, k;
  const int nlev = v.nlev;
  if (!flat_index(g.ne, nlev, e, k)) return;
  const size_t n = (size_t)g.nc * nlev;
  const size_t ie = (size_t)e * nlev + k;
  const double vne = vn[ie], vte = vt[ie];
  const int side = vne >= double(0) ? 0 : 1;
  const int cu = g.e2c[2 * e + side];
  // offset of the back-trajectory point from the upwind cell's centre, with
  // the half substep folded into the stored normal and tangent: two FMAs each
  const double* u = g.upw_s + 12 * (size_t)e + 6 * side;
  const double dx = fmat(-vne, u[2], fmat(-vte, u[4], u[0]));
  const double dy = fmat(-vne, u[3], fmat(-vte, u[5], u[1]));
  const size_t iu = (size_t)cu * nlev + k;
  double ru = rho[iu], tu = theta[iu];
  const double re = fmat(grad4[iu], dx, fmat(grad4[n + iu], dy, ru));
  const double te = fmat(grad4[2 * n + iu], dx, fmat(grad4[3 * n + iu], dy, tu));
  const int c0 = g.e2c[2 * e], c1 = g.e2c[2 * e + 1];
  const size_t i0 = (size_t)c0 * nlev + k, i1 = (size_t)c1 * nlev + k;
  // cpd theta_e d(pr)/dn with cpd folded into the edge factor cpd / d_e (and,
  // over terrain, into the stored slope)
  double h;
  const int km = k > 0 ? k - 1 : 0, kp = k + 1 < nlev ? k + 1 : nlev - 1;
  if constexpr (kTerr) {
    const size_t b0 = (size_t)c0 * nlev, b1 = (size_t)c1 * nlev;
    const double dz0 = (pex[b0 + km] - pex[b0 + kp]) * tr.inv_dzm_c[i0];
    const double dz1 = (pex[b1 + km] - pex[b1 + kp]) * tr.inv_dzm_c[i1];
    h = te * ((pex[i1] - pex[i0]) * cid64[e] - tr.ddxn_mc[ie] * (0.5 * (dz0 + dz1)));
  } else {
    h = te * ((pex[i1] - pex[i0]) * cid64[e]);
  }
  rho_e[ie] = re;
  theta_e[ie] = te;
  hpg[ie] = h;
  vn_p[ie] = vne + sc.dt_s * (ddt_vn[ie] - h);
}

// -------------------------------------------------------------------------
// A6 over steep terrain: at the listed edge levels the pressure gradient is
// taken at the edge's height, each cell's total exner (extrapolated
// perturbation plus the column's reference) interpolated there by the
// quadratic through three of its levels; the predictor's vn at those points
// follows.  Runs after sn_edge_pred, over the listed points only.
// -------------------------------------------------------------------------
template <class T>
__global__ void sn_edge_hpg_steep(GridT<T> g, VertT<T> v, ScalT<T> sc, int n, const int* __restrict__ idx,
                                  const double* __restrict__ wts, const double* __restrict__ pex,
                                  const double* __restrict__ exref_c, const double* __restrict__ cid64,
                                  const T* __restrict__ theta_e, const T* __restrict__ vn,
                                  const T* __restrict__ ddt_vn, T* __restrict__ hpg, T* __restrict__ vn_p) {
  const int i = (int)flat_thread();
  if (i >= n) return;
  const int nlev = v.nlev, ldf = v.ldf;
  const int e = idx[4 * i], k = idx[4 * i + 1];
  const int c0 = g.e2c[2 * e], c1 = g.e2c[2 * e + 1];
  const int l0 = idx[4 * i + 2], l1 = idx[4 * i + 3];
  const size_t b0 = (size_t)c0 * ldf + l0, b1 = (size_t)c1 * ldf + l1;
  const size_t r0 = (size_t)c0 * nlev + l0, r1 = (size_t)c1 * nlev + l1;
  const double* w = wts + 6 * (size_t)i;
  const size_t ie = (size_t)e * ldf + k;
  T h;
  if constexpr (kMixed<T>) {
    const df* p = reinterpret_cast<const df*>(pex);
    df s0{0.f, 0.f}, s1{0.f, 0.f};
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      s0 = s0 + to_df(w[j]) * (p[b0 + j] + to_df(exref_c[r0 + j]));
      s1 = s1 + to_df(w[3 + j]) * (p[b1 + j] + to_df(exref_c[r1 + j]));
    }
    h = theta_e[ie] * (to_float(s1 - s0) * g.cpd_inv_d[e]);
  } else {
    double s0 = 0.0, s1 = 0.0;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      s0 = fma(w[j], pex[b0 + j] + exref_c[r0 + j], s0);
      s1 = fma(w[3 + j], pex[b1 + j] + exref_c[r1 + j], s1);
    }
    h = theta_e[ie] * (T)((s1 - s0) * cid64[e]);
  }
  hpg[ie] = h;
  vn_p[ie] = vn[ie] + sc.dt_s * (ddt_vn[ie] - h);
}

// -------------------------------------------------------------------------
// A8 + A9 (corrector edges): vn corrector with time-weighted advective
// tendencies, the predictor's pressure gradient and fourth-order divergence
// damping; the increment is formed in T, the update in FP64 (in place).
// -------------------------------------------------------------------------
// Both tile shapes update every (edge, level) with sn_edge_corr_at.
template <class T>
__device__ __forceinline__ void sn_edge_corr_at(const ScalT<T>& sc, size_t iv, size_t ie, T ddamp, T d0k, T d1k,
                                                double* vn, const T* ddt_vn0, const T* ddt_vn1, const T* hpg,
                                                float* m_vn) {
  // fourth-order divergence damping: divdamp_fac Abar^2 grad_n(dd2), coefficient per edge
  const T damp = ddamp * (d1k - d0k);
  const T tend = fmat(sc.wnow_vel, ddt_vn0[ie], fmat(sc.wnew_vel, ddt_vn1[ie], -hpg[ie]));
  const T inc = fmat(sc.dt_s, tend, -damp);
  if constexpr (kMixed<T>) {
    const double vnn = vn[iv] + f2d(inc);
    vn[iv] = vnn;
    m_vn[ie] = d2f(vnn);
  } else {
    vn[iv] = vn[iv] + (double)inc;
  }
}

template <class T>
__global__ void sn_edge_corr(GridT<T> g, VertT<T> v, ScalT<T> sc, double* __restrict__ vn,
                             const T* __restrict__ ddt_vn0, const T* __restrict__ ddt_vn1,
                             const T* __restrict__ hpg, const T* __restrict__ divd2, float* __restrict__ m_vn,
                             int shape) {
  const int nlev = v.nlev, ldf = v.ldf;
  if (shape) {  // one warp per edge, its lanes over the levels
    const int e = warp_point();
    if (e >= g.ne) return;
    const int c0 = g.e2c[2 * e], c1 = g.e2c[2 * e + 1];
    const T ddamp = g.ddamp_e[e];
    const T* d0 = divd2 + (size_t)c0 * ldf;
    const T* d1 = divd2 + (size_t)c1 * ldf;
    for (int k = lane_id(); k < nlev; k += 32)
      sn_edge_corr_at(sc, (size_t)e * nlev + k, (size_t)e * ldf + k, ddamp, d0[k], d1[k], vn, ddt_vn0, ddt_vn1, hpg, m_vn);
    return;
  }
  int e, k;
  if (!flat_index(g.ne, nlev, e, k)) return;
  const int c0 = g.e2c[2 * e], c1 = g.e2c[2 * e + 1];
  sn_edge_corr_at(sc, (size_t)e * nlev + k, (size_t)e * ldf + k, g.ddamp_e[e], divd2[(size_t)c0 * ldf + k],
                  divd2[(size_t)c1 * ldf + k], vn, ddt_vn0, ddt_vn1, hpg, m_vn);
}

// -------------------------------------------------------------------------
// Cell divergence D = (1/A_c) sum_e s l_e vn_e of vn* (fourth-order damping and
// flux filter of the predictor) or vn^{n+1} (flux filter of the corrector).
// The predictor launch also updates the exner extrapolation history,
// exner_pr = exner - exner_ref (sn_edge_pred, its last reader, has completed).
// Both tile shapes evaluate every (cell, level) with the same FMAs.
// -------------------------------------------------------------------------
template <bool kTerr = false>
__global__ void sn_cell_div(GridT<double> g, VertT<double> v, const double* __restrict__ vn, double* __restrict__ divd,
                            const double* __restrict__ exner, double* __restrict__ exner_pr,
                            const double* __restrict__ exner_ref_c, int shape) {
  const int nlev = v.nlev;
  if (shape) {  // one warp per cell, its lanes over the levels
    const int c = warp_point();
    if (c >= g.nc) return;
    const int* ce = g.c2e + 3 * (size_t)c;
    const double* dvp = g.div_c + 3 * (size_t)c;
    const double dv0 = dvp[0], dv1 = dvp[1], dv2 = dvp[2];
    const double* x0 = vn + (size_t)ce[0] * nlev;
    const double* x1 = vn + (size_t)ce[1] * nlev;
    const double* x2 = vn + (size_t)ce[2] * nlev;
    for (int k = lane_id(); k < nlev; k += 32) {
      const size_t i = (size_t)c * nlev + k;
      divd[i] = fmat(dv2, x2[k], fmat(dv1, x1[k], dv0 * x0[k]));
      if (exner_pr) exner_pr[i] = exner[i] - (kTerr ? exner_ref_c[i] : v.exner_ref[k]);
    }
    return;
  }
  int c, k;
  if (!flat_index(g.nc, nlev, c, k)) return;
  const int* ce = g.c2e + 3 * (size_t)c;
  const double* dv = g.div_c + 3 * (size_t)c;
  const size_t i = (size_t)c * nlev + k;
  divd[i] = fmat(dv[2], vn[(size_t)ce[2] * nlev + k], fmat(dv[1], vn[(size_t)ce[1] * nlev + k],
                                                           dv[0] * vn[(size_t)ce[0] * nlev + k]));
  if (exner_pr) exner_pr[i] = exner[i] - (kTerr ? exner_ref_c[i] : v.exner_ref[k]);
}

// -------------------------------------------------------------------------
// FP64 mode: the same divergences from fluxes computed once per edge (the
// cell form above computes each edge's flux once for each of its two cells,
// and the FP64 mode is bound by the FP64 issue rate):
//   sn_edge_flux:    F_e = rho_e vf_e, Ft_e = F_e theta_e (edges, full levels)
//   sn_cell_fluxsum: div_m = sum s l F / A, div_t = sum s l Ft / A, over
//                    terrain with each flux times dz_e / dz_c
// -------------------------------------------------------------------------
__global__ void sn_edge_flux(GridT<double> g, VertT<double> v, const double* __restrict__ vn,
                             const double* __restrict__ divd, const double* __restrict__ rho_e,
                             const double* __restrict__ theta_e, double* __restrict__ flx_m,
                             double* __restrict__ flx_t) {
  int e, k;
  const int nlev = v.nlev;
  if (!flat_index(g.ne, nlev, e, k)) return;
  const size_t ie = (size_t)e * nlev + k;
  const int c0 = g.e2c[2 * e], c1 = g.e2c[2 * e + 1];
  const double vf = fma(g.fdiv_e[e], divd[(size_t)c1 * nlev + k] - divd[(size_t)c0 * nlev + k], vn[ie]);
  const double f = rho_e[ie] * vf;
  flx_m[ie] = f;
  flx_t[ie] = f * theta_e[ie];
}

template <bool kTerr>
__global__ void sn_cell_fluxsum(GridT<double> g, VertT<double> v, const double* __restrict__ flx_m,
                                const double* __restrict__ flx_t, double* __restrict__ div_m,
                                double* __restrict__ div_t, const double* __restrict__ fx_ratio) {
  int c, k;
  const int nlev = v.nlev;
  if (!flat_index(g.nc, nlev, c, k)) return;
  const int* ce = g.c2e + 3 * (size_t)c;
  const double* dv = g.div_c + 3 * (size_t)c;
  double dm = 0.0, dt = 0.0;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const size_t ie = (size_t)ce[j] * nlev + k;
    double fm = flx_m[ie], ft = flx_t[ie];
    if constexpr (kTerr) {
      const double r = fx_ratio[((size_t)c * 3 + j) * nlev + k];
      fm = fm * r;
      ft = ft * r;
    }
    dm = fma(dv[j], fm, dm);
    dt = fma(dv[j], ft, dt);
  }
  div_m[(size_t)c * nlev + k] = dm;
  div_t[(size_t)c * nlev + k] = dt;
}

// -------------------------------------------------------------------------
// A10 diffusion
// -------------------------------------------------------------------------
// cells: div vn; vertices: curl vn and the vertex velocity (xyz)
__global__ void diff_div_curl_uv(GridT<double> g, VertT<double> v, const double* __restrict__ vn,
                                 double* __restrict__ div_vn, double* __restrict__ zeta, double* __restrict__ uv3) {
  const int nlev = v.nlev;
  unsigned i = flat_thread();
  const unsigned ncell = (unsigned)g.nc * nlev;
  if (i < ncell) {
    int c = (int)(i / (unsigned)nlev), k = (int)(i - (unsigned)c * nlev);
    const int* ce = g.c2e + 3 * (size_t)c;
    const double* dv = g.div_c + 3 * (size_t)c;
    div_vn[(size_t)c * nlev + k] = dv[0] * vn[(size_t)ce[0] * nlev + k] + dv[1] * vn[(size_t)ce[1] * nlev + k] +
                dv[2] * vn[(size_t)ce[2] * nlev + k];
    return;
  }
  i -= ncell;
  if (i >= (size_t)g.nv * nlev) return;
  const size_t nvl = (size_t)g.nv * nlev;  // one plane of uv3
  int vx = (int)(i / (unsigned)nlev), k = (int)(i - (unsigned)vx * nlev);
  const int* ve = g.v2e + 6 * (size_t)vx;
  const double* cw = g.curl_v + 6 * (size_t)vx;
  const double* U = g.uv_w + 18 * (size_t)vx;
  double z = 0, ux = 0, uy = 0, uz = 0;
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    const double x = vn[(size_t)ve[j] * nlev + k];
    z += cw[j] * x;
    ux += U[3 * j] * x;
    uy += U[3 * j + 1] * x;
    uz += U[3 * j + 2] * x;
  }
  const size_t iv = (size_t)vx * nlev + k;
  zeta[iv] = z;
  uv3[iv] = ux;
  uv3[nvl + iv] = uy;
  uv3[2 * nvl + iv] = uz;
}

// edges: Smagorinsky coefficient (times dtime) and the vector Laplacian of vn.
// Bound by the FP64 pipe: the coefficients carry every factor of the tension
// and the shear, and the square root takes two FP64 operations: 26 a
// point-level instead of 35, 122880 edges of 90 levels 733 -> 554 us.
__global__ void diff_edge_smag(GridT<double> g, VertT<double> v, const double* __restrict__ div_vn,
                               const double* __restrict__ zeta, const double* __restrict__ uv3, double* __restrict__ nu,
                               double* __restrict__ lap) {
  int e, k;
  const int nlev = v.nlev;
  if (!flat_index(g.ne, nlev, e, k)) return;
  const size_t nvl = (size_t)g.nv * nlev;
  const int* dm = g.e2c2v + 4 * (size_t)e;
  const size_t im = (size_t)dm[0] * nlev + k, ip = (size_t)dm[1] * nlev + k;
  const size_t i2 = (size_t)dm[2] * nlev + k, i3 = (size_t)dm[3] * nlev + k;
  const double dtx = uv3[ip] - uv3[im], dty = uv3[nvl + ip] - uv3[nvl + im];
  const double dtz = uv3[2 * nvl + ip] - uv3[2 * nvl + im];
  const double dnx = uv3[i3] - uv3[i2], dny = uv3[nvl + i3] - uv3[nvl + i2];
  const double dnz = uv3[2 * nvl + i3] - uv3[2 * nvl + i2];
  const double* q = g.smag_c + 12 * (size_t)e;
  const double tension =
      fma(dnx, q[0], fma(dny, q[1], fma(dnz, q[2], -fma(dtx, q[3], fma(dty, q[4], dtz * q[5])))));
  const double shear = fma(dtx, q[6], fma(dty, q[7], fma(dtz, q[8], fma(dnx, q[9], fma(dny, q[10], dnz * q[11])))));
  const size_t ie = (size_t)e * nlev + k;
  const double a = sqrt2(fma(tension, tension, shear * shear));
  nu[ie] = g.smag_a[e] < 0.0 ? -a : a;
  const int c0 = g.e2c[2 * e], c1 = g.e2c[2 * e + 1];
  lap[ie] = (div_vn[(size_t)c1 * nlev + k] - div_vn[(size_t)c0 * nlev + k]) * g.inv_d[e] -
            (zeta[ip] - zeta[im]) * g.inv_l[e];
}

// cells (half-level range): div of lap vn, cell Laplacian of w, theta increment;
// vertices: curl of lap vn
__global__ void diff_second(GridT<double> g, VertT<double> v, ScalT<double> sc, const double* __restrict__ lap,
                            const double* __restrict__ nu, const double* __restrict__ w,
                            const double* __restrict__ theta, double* __restrict__ div_l, double* __restrict__ lap_w,
                            double* __restrict__ dtheta, double* __restrict__ curl_l,
                            const double* __restrict__ tenh_ex) {
  const int nlev = v.nlev, nlevp = nlev + 1;
  unsigned i = flat_thread();
  const unsigned ncell = (unsigned)g.nc * nlevp;
  if (i < ncell) {
    int c = (int)(i / (unsigned)nlevp), k = (int)(i - (unsigned)c * nlevp);
    const int* ce = g.c2e + 3 * (size_t)c;
    const int* cc = g.c2e2c + 3 * (size_t)c;
    const double* L = g.lap_c + 3 * (size_t)c;
    const double wc = w[(size_t)c * nlevp + k];
    double lw = L[0] * (w[(size_t)cc[0] * nlevp + k] - wc);
    lw += L[1] * (w[(size_t)cc[1] * nlevp + k] - wc);
    lw += L[2] * (w[(size_t)cc[2] * nlevp + k] - wc);
    lap_w[(size_t)c * nlevp + k] = lw;
    if (k < nlev) {
      const double* dv = g.div_c + 3 * (size_t)c;
      const size_t ic = (size_t)c * nlev + k;
      div_l[ic] = dv[0] * lap[(size_t)ce[0] * nlev + k] + dv[1] * lap[(size_t)ce[1] * nlev + k] +
                  dv[2] * lap[(size_t)ce[2] * nlev + k];
      if (sc.hdiff_temp) {
        const double tc = theta[ic];
        double n0 = nu[(size_t)ce[0] * nlev + k], n1 = nu[(size_t)ce[1] * nlev + k], n2 = nu[(size_t)ce[2] * nlev + k];
        if (k >= nlev - sc.tenh_levels) {
          // enhanced near-surface temperature diffusion: the edge coefficient
          // raised by fac A_e / dtime max(e_c, e_nbr) (here all times dtime)
          const double ex = tenh_ex[ic];
          n0 += g.tenh_a[ce[0]] * max(ex, tenh_ex[(size_t)cc[0] * nlev + k]);
          n1 += g.tenh_a[ce[1]] * max(ex, tenh_ex[(size_t)cc[1] * nlev + k]);
          n2 += g.tenh_a[ce[2]] * max(ex, tenh_ex[(size_t)cc[2] * nlev + k]);
        }
        double f = L[0] * n0 * (theta[(size_t)cc[0] * nlev + k] - tc);
        f += L[1] * n1 * (theta[(size_t)cc[1] * nlev + k] - tc);
        f += L[2] * n2 * (theta[(size_t)cc[2] * nlev + k] - tc);
        dtheta[ic] = f;
      }
    }
    return;
  }
  i -= ncell;
  if (i >= (unsigned)g.nv * nlev) return;
  int vx = (int)(i / (unsigned)nlev), k = (int)(i - (unsigned)vx * nlev);
  const int* ve = g.v2e + 6 * (size_t)vx;
  const double* cw = g.curl_v + 6 * (size_t)vx;
  double z = 0;
#pragma unroll
  for (int j = 0; j < 6; ++j) z += cw[j] * lap[(size_t)ve[j] * nlev + k];
  curl_l[(size_t)vx * nlev + k] = z;
}

// cells, the lowest tenh_levels levels: the excess factor of the enhanced
// temperature diffusion, e_c = min(1, (|theta_c - mean of the three neighbours|
// - thresh) / thresh) where above the threshold, else 0 (theta as the stencil
// views it: the FP64 state, or the mixed mode's perturbation from a per-level
// offset, which the difference does not see)
template <class T>
__global__ void diff_tenh_excess(GridT<T> g, VertT<T> v, ScalT<T> sc, const T* __restrict__ theta,
                                 T* __restrict__ ex) {
  const int nlev = v.nlev, ldf = v.ldf, nl = sc.tenh_levels;
  const unsigned i = flat_thread();
  if (i >= (unsigned)g.nc * (unsigned)nl) return;
  const int c = (int)(i / (unsigned)nl), k = nlev - nl + (int)(i - (unsigned)c * (unsigned)nl);
  const int* cc = g.c2e2c + 3 * (size_t)c;
  const size_t ic = (size_t)c * ldf + k;
  const T nbr = (theta[(size_t)cc[0] * ldf + k] + theta[(size_t)cc[1] * ldf + k] + theta[(size_t)cc[2] * ldf + k]) /
                T(3);
  const T x = (abs(theta[ic] - nbr) - sc.tenh_thresh) / sc.tenh_thresh;
  ex[ic] = x < T(0) ? T(0) : (x > T(1) ? T(1) : x);
}

// edges: vn update (FP64, in place)
__global__ void diff_edge_update(GridT<double> g, VertT<double> v, ScalT<double> sc, double* __restrict__ vn,
                                 const double* __restrict__ nu, const double* __restrict__ lap,
                                 const double* __restrict__ div_l, const double* __restrict__ curl_l) {
  int e, k;
  const int nlev = v.nlev;
  if (!flat_index(g.ne, nlev, e, k)) return;
  const size_t ie = (size_t)e * nlev + k;
  const int c0 = g.e2c[2 * e], c1 = g.e2c[2 * e + 1];
  const int vm = g.e2v[2 * e], vp = g.e2v[2 * e + 1];
  const double lap2 = (div_l[(size_t)c1 * nlev + k] - div_l[(size_t)c0 * nlev + k]) * g.inv_d[e] -
                 (curl_l[(size_t)vp * nlev + k] - curl_l[(size_t)vm * nlev + k]) * g.inv_l[e];
  const double inc = nu[ie] * lap[ie] - g.k4_a[e] * lap2;
  vn[ie] = vn[ie] + inc;
}

// cells (half-level range): w fourth-order diffusion, theta/exner update (FP64,
// in place).  FP64 operations bound it: 12 a point-level with the reciprocal of
// theta instead of 19 with the division, 81920 cells of 90 levels 276 -> 183 us.
__global__ void diff_cell_update(GridT<double> g, VertT<double> v, ScalT<double> sc, double rd_o_cvd, StateView st,
                                 const double* __restrict__ lap_w, const double* __restrict__ dtheta) {
  int c, k;
  const int nlev = v.nlev, nlevp = nlev + 1;
  if (!flat_index(g.nc, nlevp, c, k)) return;
  if (k > 0 && k < nlev) {
    const int* cc = g.c2e2c + 3 * (size_t)c;
    const double* L = g.lap_c + 3 * (size_t)c;
    const double lc = lap_w[(size_t)c * nlevp + k];
    double l2 = L[0] * (lap_w[(size_t)cc[0] * nlevp + k] - lc);
    l2 += L[1] * (lap_w[(size_t)cc[1] * nlevp + k] - lc);
    l2 += L[2] * (lap_w[(size_t)cc[2] * nlevp + k] - lc);
    const size_t iw = (size_t)c * nlevp + k;
    st.w[iw] = st.w[iw] - g.k4w_c[c] * l2;
  }
  if (k < nlev && sc.hdiff_temp) {
    const size_t ic = (size_t)c * nlev + k;
    const double th = st.theta_v[ic], dth = dtheta[ic], ex = st.exner[ic];
    st.theta_v[ic] = th + dth;
    st.exner[ic] = fma(ex, (rd_o_cvd * dth) * rcp(th), ex);
  }
}

}  // namespace

// -------------------------------------------------------------------------
// launch sequences
// -------------------------------------------------------------------------
namespace {
// whether rows of nlev FP64 values of these arrays can be read two at a time
bool aligned_pairs(int nlev, std::initializer_list<const double*> arrays) {
  size_t bits = 0;
  for (const double* p : arrays) bits |= reinterpret_cast<size_t>(p);
  return nlev % 2 == 0 && bits % 16 == 0;
}
}  // namespace

template <class T>
void launch_velocity_tendencies(const Ctx<T>& x, const T* vn, const T* w, T* ddt_vn, T* ddt_w, const T* divd,
                                T* divd2, cudaStream_t s, const int* threads, T* wcc, const int* shapes) {
  const GridT<T>& g = x.g;
  const VertT<T>& v = x.v;
  const WorkT<T>& wk = x.w;
  const TerrT<T>& tr = x.tr;
  const int nlev = v.nlev, nlevp = nlev + 1;
  const bool terr = tr.wgt_e != nullptr && wcc != nullptr;
  if constexpr (kMixed<T>) {
    if (x.vp.n_patches > 0 && !terr) {  // rows A1-A4 in one launch
      const VaPatchT& pt = x.vp;
      const size_t smem =
          va_fused_smem_floats(pt.max_e0, pt.max_e1, pt.max_c3, pt.max_c0, pt.max_v3, pt.max_e4) * sizeof(float);
      ICON_CHAIN_SMEM("va_fused_f32", (unsigned)pt.n_patches, kVaThreads, smem, s, va_fused, g, v, pt, vn, w, wk.vt,
                       ddt_vn, ddt_w, divd, divd2);
      return;
    }
    // four levels per thread
    const long long nqf = quads_full(nlev), nqh = quads_half(nlev);
    T* const q_wcc = terr ? wcc : nullptr;
    ICON_CHAIN("va_edge_pre_f32", blocks_for(g.ne * nqf, TH(0)), TH(0), s, va_edge_pre_q, g, v, vn, wk.vt, wk.ekin_e,
                wk.vn_ie, terr ? tr.wgt_e : nullptr);
    if (terr)
      ICON_CHAIN("va_concorr_f32", blocks_for(g.nc * nqh, TH(14)), TH(14), s, va_concorr_q, g, v, tr, wk.vn_ie,
                  wk.vt, wcc);
    ICON_CHAIN("va_cell_vert_f32", blocks_for(g.nc * nqf + g.nv * nqh, TH(1)), TH(1), s, va_cell_vert_q, g, v, vn, w,
                wk.ekin_e, wk.ekin_c, divd, divd2, wk.zeta, wk.w_v, wk.wq, q_wcc);
    const char* const nm_tend = terr ? "va_edge_tend_terrain_f32" : "va_edge_tend_f32";
    const char* const nm_w = terr ? "va_cell_w_terrain_f32" : "va_cell_w_f32";
    ICON_CHAIN(nm_tend, blocks_for(g.ne * nqh, TH(2)), TH(2), s, (terr ? va_edge_tend_q<true> : va_edge_tend_q<false>),
                g, v, wk.vn_ie, w, wk.vt, wk.ekin_c, wk.zeta, wk.w_v, ddt_vn, wk.gw_e, tr, wk.wq);
    ICON_CHAIN(nm_w, blocks_for(g.nc * nqh, TH(3)), TH(3), s, (terr ? va_cell_w_q<true> : va_cell_w_q<false>), g, v,
                w, wk.gw_e, ddt_w, tr, q_wcc);
  } else {
    ICON_CHAIN("va_edge_pre", blocks_by_shape(SH(0), g.ne, nlev, TH(0)), TH(0), s, va_edge_pre, g, v, vn, wk.vt,
                wk.ekin_e, wk.vn_ie, terr ? tr.wgt_e : nullptr, SH(0));
    if (terr)
      ICON_CHAIN("va_concorr", blocks_for((long long)g.nc * nlevp, TH(14)), TH(14), s, va_concorr, g, v, tr,
                  wk.vn_ie, wk.vt, wcc);
    const long long n2 = (long long)g.nc * nlev + (long long)g.nv * nlevp;
    ICON_CHAIN("va_cell_vert", blocks_for(n2, TH(1)), TH(1), s, va_cell_vert, g, v, vn, w, wk.ekin_e, wk.ekin_c, divd,
                divd2, wk.zeta, wk.w_v, wk.wq, terr ? (const T*)wcc : nullptr);
    if (terr) {
      ICON_CHAIN("va_edge_tend_terrain", blocks_for((long long)g.ne * nlevp, TH(2)), TH(2), s, va_edge_tend<true>, g,
                  v, wk.vn_ie, w, wk.vt, wk.ekin_c, wk.zeta, wk.w_v, ddt_vn, wk.gw_e, tr, (const T*)wk.wq);
      ICON_CHAIN("va_cell_w_terrain", blocks_by_shape(SH(3), g.nc, nlevp, TH(3)), TH(3), s, va_cell_w<true>, g, v, w,
                  wk.gw_e, ddt_w, tr, wcc, SH(3));
    } else {
      ICON_CHAIN("va_edge_tend", blocks_for((long long)g.ne * nlevp, TH(2)), TH(2), s, va_edge_tend<false>, g, v,
                  wk.vn_ie, w, wk.vt, wk.ekin_c, wk.zeta, wk.w_v, ddt_vn, wk.gw_e, tr, (const T*)wk.wq);
      ICON_CHAIN("va_cell_w", blocks_by_shape(SH(3), g.nc, nlevp, TH(3)), TH(3), s, va_cell_w<false>, g, v, w,
                  wk.gw_e, ddt_w, tr, wcc, SH(3));
    }
  }
}

// Flux divergences of the mass and theta fluxes of the velocity vn (with the
// flux filter): the mixed mode sums FP32 fluxes per cell in double-word
// arithmetic; the FP64 mode computes each edge's fluxes once, then sums them.
template <class T, bool kTerr>
void launch_fluxdiv(const Engine& en, const Ctx<T>& x, const T* vn, const char* name, cudaStream_t s) {
  const int* threads = en.threads;
  const GridT<T>& g = x.g;
  const VertT<T>& v = x.v;
  const WorkT<T>& wk = x.w;
  const int nlev = v.nlev;
  if constexpr (kMixed<T>) {
    ICON_CHAIN(name, blocks_for((long long)g.nc * quads_full(nlev), TH(7)), TH(7), s, sn_cell_fluxdiv_q<kTerr>, g, v,
                vn, wk.divd, wk.rho_e, wk.theta_e, reinterpret_cast<df*>(en.wk.div_m),
                reinterpret_cast<df*>(en.wk.div_t), x.tr.fx_ratio);
  } else {
    ICON_CHAIN("sn_edge_flux", blocks_for((long long)g.ne * nlev, TH(15)), TH(15), s, sn_edge_flux, g, v, vn,
                wk.divd, wk.rho_e, wk.theta_e, wk.flx_m, wk.flx_t);
    ICON_CHAIN(kTerr ? "sn_cell_fluxsum_terrain" : "sn_cell_fluxsum", blocks_for((long long)g.nc * nlev, TH(7)),
                TH(7), s, (sn_cell_fluxsum<kTerr>), g, v, wk.flx_m, wk.flx_t, en.wk.div_m, en.wk.div_t,
                x.tr.fx_ratio);
  }
}

// Rows A5-A9 of one substep; kTerr: the terrain forms, with the contravariant
// corrections of the predictor's and the corrector's winds in x.tr.wcc0/wcc1.
// s waits for event e: as an external event node when s is being captured
// into a graph (the wait then happens at every launch of the graph), else as
// a plain stream wait
void stream_wait_io(cudaStream_t s, cudaEvent_t e) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  cudaStreamIsCapturing(s, &cs);
  cudaStreamWaitEvent(s, e, cs == cudaStreamCaptureStatusActive ? cudaEventWaitExternal : 0);
}
void stream_record_io(cudaStream_t s, cudaEvent_t e) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  cudaStreamIsCapturing(s, &cs);
  cudaEventRecordWithFlags(e, s, cs == cudaStreamCaptureStatusActive ? cudaEventRecordExternal : 0);
}

template <class T, bool kTerr>
void substep_impl(const Engine& en, const Ctx<T>& x, const StateView& st, cudaStream_t s) {
  const int* threads = en.threads;
  const int* shapes = en.shape;
  const GridT<T>& g = x.g;
  const VertT<T>& v = x.v;
  const WorkT<T>& wk = x.w;
  const TerrT<T>& tr = x.tr;
  const Mirrors& m = en.m;
  const int nlev = v.nlev;
  const long long nce = (long long)g.nc * nlev, nee = (long long)g.ne * nlev, nqf = quads_full(nlev);
  const double* ex_ref_c = en.v.exner_ref_c;
  // the caller's FP64 rows in aligned pairs of levels (the quad kernels)
  const bool pairs = aligned_pairs(nlev, {st.exner, st.exner_pr});
  // stencil views of the state: the FP64 state itself, or the FP32 mirrors
  const T *s_vn, *s_w, *s_rho, *s_th, *s_wp;
  if constexpr (kMixed<T>) {
    s_vn = m.vn, s_w = m.w, s_rho = m.rho, s_th = m.th, s_wp = m.w_p;
  } else {
    s_vn = st.vn, s_w = st.w, s_rho = st.rho, s_th = st.theta_v, s_wp = en.wk.w_p;
  }
  const char* nm_grad = kTerr ? kname<T>("sn_cell_grad_terrain", "sn_cell_grad_terrain_f32")
                              : kname<T>("sn_cell_grad", "sn_cell_grad_f32");
  const char* nm_pred = kTerr ? kname<T>("sn_edge_pred_terrain", "sn_edge_pred_terrain_f32")
                              : kname<T>("sn_edge_pred", "sn_edge_pred_f32");
  const char* nm_div = kTerr ? kname<T>("sn_cell_div_terrain", "sn_cell_div_terrain_f32")
                             : kname<T>("sn_cell_div", "sn_cell_div_f32");
  const char* nm_flx = kTerr ? kname<T>("sn_cell_fluxdiv_terrain", "sn_cell_fluxdiv_terrain_f32")
                             : kname<T>("sn_cell_fluxdiv", "sn_cell_fluxdiv_f32");
  // ---------------- predictor ----------------
  launch_velocity_tendencies<T>(x, s_vn, s_w, wk.ddt_vn0, wk.ddt_w0, nullptr, nullptr, s, threads,
                                kTerr ? tr.wcc0 : nullptr, shapes);
  if (en.io_wait) stream_wait_io(s, en.io_wait);  // rho, theta_v, exner, exner_pr from here on
  if constexpr (kMixed<T>) {
    ICON_CHAIN(nm_grad, blocks_for(g.nc * nqf, TH(4)), TH(4), s, sn_cell_grad_q<kTerr>, g, v, s_rho, s_th, wk.grad4,
                st.exner, st.exner_pr, en.sc.exfac, reinterpret_cast<df*>(en.wk.pex), ex_ref_c, pairs);
    ICON_CHAIN(nm_pred, blocks_for(g.ne * nqf, TH(5)), TH(5), s, sn_edge_pred_q<kTerr>, g, v, x.s, s_vn, wk.vt,
                wk.ddt_vn0, s_rho, s_th, reinterpret_cast<const df*>(en.wk.pex), wk.grad4, wk.rho_e, wk.theta_e,
                wk.hpg, wk.vn_p, tr);
  } else {
    ICON_CHAIN(nm_grad, blocks_for(nce, TH(4)), TH(4), s, sn_cell_grad<kTerr>, g, v, s_rho, s_th, wk.grad4, st.exner,
                st.exner_pr, en.sc.exfac, en.wk.pex, ex_ref_c);
    ICON_CHAIN(nm_pred, blocks_for(nee, TH(5)), TH(5), s, sn_edge_pred<kTerr>, g, v, x.s, s_vn, wk.vt, wk.ddt_vn0,
                s_rho, s_th, en.wk.pex, en.g64.cpd_inv_d, wk.grad4, wk.rho_e, wk.theta_e, wk.hpg, wk.vn_p, tr);
  }
  if (kTerr && en.v.n_steep > 0)
    ICON_CHAIN(kname<T>("sn_edge_hpg_steep", "sn_edge_hpg_steep_f32"), blocks_for(en.v.n_steep, 128), 128, s,
                sn_edge_hpg_steep<T>, g, v, x.s, en.v.n_steep, en.v.steep_idx, en.v.steep_w, en.wk.pex,
                en.v.exner_ref_c, en.g64.cpd_inv_d, wk.theta_e, s_vn, wk.ddt_vn0, wk.hpg, wk.vn_p);
  // divergence of a velocity field; the predictor's call also updates the exner history
  auto cell_div = [&](const T* vn, double* exner_pr) {
    if constexpr (kMixed<T>)
      ICON_CHAIN(nm_div, blocks_for(g.nc * nqf, TH(6)), TH(6), s, sn_cell_div_q<kTerr>, g, v, vn, wk.divd, st.exner,
                  exner_pr, ex_ref_c, pairs);
    else
      ICON_CHAIN(nm_div, blocks_by_shape(SH(6), g.nc, nlev, TH(6)), TH(6), s, sn_cell_div<kTerr>, g, v, vn, wk.divd,
                  st.exner, exner_pr, ex_ref_c, SH(6));
  };
  cell_div(wk.vn_p, st.exner_pr);
  launch_fluxdiv<T, kTerr>(en, x, wk.vn_p, nm_flx, s);
  if constexpr (kTerr)
    launch_column_terrain<T>(en, 0, st, wk.ddt_w0, wk.ddt_w1, tr.wcc0, s);
  else
    launch_column<T>(en, 0, st, wk.ddt_w0, wk.ddt_w1, s);
  // ---------------- corrector ----------------
  launch_velocity_tendencies<T>(x, wk.vn_p, s_wp, wk.ddt_vn1, wk.ddt_w1, wk.divd, wk.divd2, s, threads,
                                kTerr ? tr.wcc1 : nullptr, shapes);
  ICON_CHAIN(kname<T>("sn_edge_corr", "sn_edge_corr_f32"), blocks_by_shape(SH(8), g.ne, nlev, TH(8)), TH(8), s,
              sn_edge_corr<T>, g, v, x.s, st.vn, wk.ddt_vn0, wk.ddt_vn1, wk.hpg, wk.divd2, m.vn, SH(8));
  const T* vn_new = kMixed<T> ? (const T*)m.vn : (const T*)st.vn;
  cell_div(vn_new, nullptr);
  launch_fluxdiv<T, kTerr>(en, x, vn_new, nm_flx, s);
  if constexpr (kTerr)
    launch_column_terrain<T>(en, 1, st, wk.ddt_w0, wk.ddt_w1, tr.wcc1, s);
  else
    launch_column<T>(en, 1, st, wk.ddt_w0, wk.ddt_w1, s);
}

template <class T>
void launch_substep(const Engine& en, const Ctx<T>& x, const StateView& st, cudaStream_t s) {
  if (en.terrain)
    substep_impl<T, true>(en, x, st, s);
  else
    substep_impl<T, false>(en, x, st, s);
}

template <class T>
void launch_diffusion(const Engine& en, const Ctx<T>& x, const StateView& st, cudaStream_t s) {
  const int* threads = en.threads;
  const GridT<T>& g = x.g;
  const VertT<T>& v = x.v;
  const WorkT<T>& wk = x.w;
  const Mirrors& m = en.m;
  const int nlev = v.nlev, nlevp = nlev + 1;
  const T *s_vn, *s_w, *s_th;
  if constexpr (kMixed<T>) {
    s_vn = m.vn, s_w = m.w, s_th = m.th;
  } else {
    s_vn = st.vn, s_w = st.w, s_th = st.theta_v;
  }
  const long long nqf = quads_full(nlev), nqh = quads_half(nlev);
  const long long n1 = (long long)(g.nc + g.nv) * nlev;
  const long long n3 = (long long)g.nc * nlevp + (long long)g.nv * nlev;
  if constexpr (kMixed<T>) {  // four levels per thread
    ICON_CHAIN("diff_div_curl_uv_f32", blocks_for((g.nc + g.nv) * nqf, TH(9)), TH(9), s, diff_div_curl_uv_q, g, v,
                s_vn, wk.div_vn, wk.zeta, wk.uv3);
    ICON_CHAIN("diff_edge_smag_f32", blocks_for(g.ne * nqf, TH(10)), TH(10), s, diff_edge_smag_q, g, v, wk.div_vn,
                wk.zeta, wk.uv3, wk.nu, wk.lap_vn);
  } else {
    ICON_CHAIN("diff_div_curl_uv", blocks_for(n1, TH(9)), TH(9), s, diff_div_curl_uv, g, v, s_vn, wk.div_vn, wk.zeta,
                wk.uv3);
    ICON_CHAIN("diff_edge_smag", blocks_for((long long)g.ne * nlev, TH(10)), TH(10), s, diff_edge_smag, g, v,
                wk.div_vn, wk.zeta, wk.uv3, wk.nu, wk.lap_vn);
  }
  if (x.s.tenh_levels > 0 && x.s.hdiff_temp)
    ICON_CHAIN(kname<T>("diff_tenh_excess", "diff_tenh_excess_f32"),
                blocks_for((long long)g.nc * x.s.tenh_levels, kThreads), kThreads, s, diff_tenh_excess<T>, g, v, x.s,
                s_th, wk.tenh_ex);
  if constexpr (kMixed<T>) {
    ICON_CHAIN("diff_second_f32", blocks_for(g.nc * nqh + g.nv * nqf, TH(11)), TH(11), s, diff_second_q, g, v, x.s,
                wk.lap_vn, wk.nu, s_w, s_th, wk.div_l, wk.lap_w, wk.dtheta, wk.curl_l, wk.tenh_ex);
    ICON_CHAIN("diff_edge_update_f32", blocks_for(g.ne * nqf, TH(12)), TH(12), s, diff_edge_update_q, g, v, x.s,
                st.vn, wk.nu, wk.lap_vn, wk.div_l, wk.curl_l, m.vn, aligned_pairs(nlev, {st.vn}));
    ICON_CHAIN("diff_cell_update_f32", blocks_for(g.nc * nqh, TH(13)), TH(13), s, diff_cell_update_q, g, v, x.s,
                en.v.theta_ref, en.sc.rd_o_cvd, st, wk.lap_w, wk.dtheta, m,
                aligned_pairs(nlev, {st.theta_v, st.exner}));
  } else {
    ICON_CHAIN("diff_second", blocks_for(n3, TH(11)), TH(11), s, diff_second, g, v, x.s, wk.lap_vn, wk.nu, s_w, s_th,
                wk.div_l, wk.lap_w, wk.dtheta, wk.curl_l, wk.tenh_ex);
    ICON_CHAIN("diff_edge_update", blocks_for((long long)g.ne * nlev, TH(12)), TH(12), s, diff_edge_update, g, v,
                x.s, st.vn, wk.nu, wk.lap_vn, wk.div_l, wk.curl_l);
    ICON_CHAIN("diff_cell_update", blocks_for((long long)g.nc * nlevp, TH(13)), TH(13), s, diff_cell_update, g, v,
                x.s, en.sc.rd_o_cvd, st, wk.lap_w, wk.dtheta);
  }
}

namespace {
__global__ void fill_kernel(double* p, size_t n, double v) {
  const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (i < n) p[i] = v;
}
}  // namespace

cudaError_t init_va_fused(const VaPatchT& pt) {
  const size_t bytes = va_fused_smem_floats(pt.max_e0, pt.max_e1, pt.max_c3, pt.max_c0, pt.max_v3, pt.max_e4) * sizeof(float);
  if (bytes > 227 * 1024) return cudaErrorInvalidValue;
  return cudaFuncSetAttribute(va_fused, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

void launch_fill(double* p, size_t n, double v, cudaStream_t s) {
  fill_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(p, n, v);
}

const char* const kStencilNames[kNumStencils] = {
    "va_edge_pre", "va_cell_vert", "va_edge_tend", "va_cell_w", "sn_cell_grad", "sn_edge_pred", "sn_cell_div",
    "sn_cell_fluxdiv", "sn_edge_corr", "diff_div_curl_uv", "diff_edge_smag", "diff_second", "diff_edge_update",
    "diff_cell_update", "va_concorr", "sn_edge_flux"};

void launch_gradient_frame(const Engine& en, double* f, cudaStream_t s) {
  const int nlev = en.v.nlev;
  gradient_frame<<<blocks_for((long long)en.g64.nc * nlev, kThreads), kThreads, 0, s>>>(en.g64, nlev, f);
}

void launch_refresh_mirrors(const Engine& en, const StateView& st, cudaStream_t s) {
  const int nlev = en.v.nlev;
  const long long n = (long long)en.g64.ne * quads_full(nlev) + (long long)en.g64.nc * quads_half(nlev);
  ICON_CHAIN("mx_refresh", blocks_for(n, kThreads), kThreads, s, mx_refresh, en.g64.ne, en.g64.nc, en.c32.v,
              en.v.theta_ref, en.rho_ref64, st, en.m, aligned_pairs(nlev, {st.vn, st.rho, st.theta_v}));
}

template void launch_velocity_tendencies<double>(const Ctx<double>&, const double*, const double*, double*, double*,
                                                 const double*, double*, cudaStream_t, const int*, double*,
                                                 const int*);
template void launch_substep<double>(const Engine&, const Ctx<double>&, const StateView&, cudaStream_t);
template void launch_substep<float>(const Engine&, const Ctx<float>&, const StateView&, cudaStream_t);
template void launch_diffusion<double>(const Engine&, const Ctx<double>&, const StateView&, cudaStream_t);
template void launch_diffusion<float>(const Engine&, const Ctx<float>&, const StateView&, cudaStream_t);

}  // namespace icon
