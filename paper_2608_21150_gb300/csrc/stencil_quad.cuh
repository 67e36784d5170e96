// FP32 stencil kernels of the mixed modes, four consecutive levels per thread
// (rows A1-A6, A8, A10).  Included by kernels_stencil.cu.
//
// These kernels wait on gathers: with one thread per (point, level) a thread
// loads its neighbour indices, then some twenty 4-byte values, and DRAM ran at
// 32-56 % with the loads as the top stall.  The FP32 rows are padded to ld, a
// multiple of four floats, so a thread takes four levels of every field with
// one 16-byte load: a quarter of the index loads and instructions and four
// times the bytes in flight per load.  Pad entries hold whatever the
// arithmetic makes of pads; no level reads them.  Every level's expression is
// rounded as in the one-level form, so the bits are the same.
//
// At 327680 cells, 491520 edges and 90 levels, one level per thread -> a quad
// (us a launch): va_edge_pre 197 -> 125, va_cell_vert 331 -> 179, va_edge_tend
// 404 -> 234, va_cell_w 119 -> 71, sn_cell_grad 308 -> 238, sn_edge_pred
// 478 -> 371, sn_cell_div 131 -> 88, sn_cell_fluxdiv 336 -> 228, mx_refresh
// 382 -> 234, diff_div_curl_uv 262 -> 150, diff_edge_smag 402 -> 254,
// diff_second 369 -> 241, diff_edge_update 301 -> 215, diff_cell_update
// 405 -> 355; at 81920 cells over terrain va_concorr 80 -> 56.  DRAM bounds
// what is left; mx_refresh and the updates move the FP64 state, in pairs where
// the caller's rows allow it.
#pragma once

namespace icon {
namespace {

__device__ __forceinline__ void ld4(float (&a)[4], const float* p) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  a[0] = v.x, a[1] = v.y, a[2] = v.z, a[3] = v.w;
}
__device__ __forceinline__ void st4(float* p, const float (&a)[4]) {
  *reinterpret_cast<float4*>(p) = make_float4(a[0], a[1], a[2], a[3]);
}
// four double-word pairs of a row padded to ld
__device__ __forceinline__ void ld4(df (&a)[4], const df* p) {
  const float4 x = reinterpret_cast<const float4*>(p)[0], y = reinterpret_cast<const float4*>(p)[1];
  a[0] = {x.x, x.y}, a[1] = {x.z, x.w}, a[2] = {y.x, y.y}, a[3] = {y.z, y.w};
}
__device__ __forceinline__ void st4(df* p, const df (&a)[4]) {
  reinterpret_cast<float4*>(p)[0] = make_float4(a[0].hi, a[0].lo, a[1].hi, a[1].lo);
  reinterpret_cast<float4*>(p)[1] = make_float4(a[2].hi, a[2].lo, a[3].hi, a[3].lo);
}

// quads of the full levels 0 .. nlev-1 and of the half levels 0 .. nlev
__host__ __device__ inline int quads_full(int nlev) { return (nlev + 3) / 4; }
__host__ __device__ inline int quads_half(int nlev) { return nlev / 4 + 1; }

// point h and first level k of this thread's quad
__device__ __forceinline__ bool quad_index(int n_h, int nq, int& h, int& k) {
  int q;
  if (!flat_index(n_h, nq, h, q)) return false;
  k = 4 * q;
  return true;
}

// A1, as va_edge_pre
__global__ void va_edge_pre_q(GridT<float> g, VertT<float> v, const float* __restrict__ vn, float* __restrict__ vt,
                              float* __restrict__ ekin, float* __restrict__ vn_ie, const float* __restrict__ wgt_e) {
  int e, k;
  const int nlev = v.nlev, ld = v.ldf;
  if (!quad_index(g.ne, quads_full(nlev), e, k)) return;
  const int4 q = *reinterpret_cast<const int4*>(g.e2c2e + 4 * (size_t)e);
  const float* w = g.vt_w + 5 * (size_t)e;
  const size_t i = (size_t)e * ld + k;
  float x0[4], x1[4], x2[4], x3[4], x4[4], wg[4];
  ld4(x0, vn + i);
  ld4(x1, vn + (size_t)q.x * ld + k);
  ld4(x2, vn + (size_t)q.y * ld + k);
  ld4(x3, vn + (size_t)q.z * ld + k);
  ld4(x4, vn + (size_t)q.w * ld + k);
  ld4(wg, wgt_e ? wgt_e + i : v.wgt + k);
  const float xm = k > 0 ? vn[i - 1] : 0.0f;
  const float w0 = w[0], w1 = w[1], w2 = w[2], w3 = w[3], w4 = w[4];
  float o_vt[4], o_k[4], o_ie[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float vne = x0[j];
    float t = w0 * vne;
    t = fmat(w1, x1[j], t);
    t = fmat(w2, x2[j], t);
    t = fmat(w3, x3[j], t);
    t = fmat(w4, x4[j], t);
    o_vt[j] = t;
    o_k[j] = fmat(vne, vne, t * t);
    const float up = j == 0 ? xm : x0[j > 0 ? j - 1 : 0];
    o_ie[j] = k + j == 0 ? vne : k + j >= nlev ? up : fmat(wg[j], up - vne, vne);
  }
  st4(vt + i, o_vt);
  st4(ekin + i, o_k);
  st4(vn_ie + i, o_ie);
  if (k + 4 == nlev) vn_ie[i + 4] = x0[3];  // the ground's half level opens a quad of its own
}

// A2, as va_cell_vert: one launch over the cells' full-level and the
// vertices' half-level quads
__global__ void va_cell_vert_q(GridT<float> g, VertT<float> v, const float* __restrict__ vn,
                               const float* __restrict__ w, const float* __restrict__ ekin_e,
                               float* __restrict__ ekin_c, const float* __restrict__ divd, float* __restrict__ divd2,
                               float* __restrict__ zeta, float* __restrict__ w_v, float* __restrict__ wq,
                               const float* __restrict__ wcc) {
  const int nlev = v.nlev, ld = v.ldf, nqf = quads_full(nlev), nqh = quads_half(nlev);
  unsigned t = flat_thread();
  const unsigned ncell = (unsigned)g.nc * nqf;
  if (t < ncell) {
    const int c = (int)(t / (unsigned)nqf), k = 4 * (int)(t - (unsigned)c * nqf);
    const int* ce = g.c2e + 3 * (size_t)c;
    const float* q = g.e2c_w + 3 * (size_t)c;
    const size_t i = (size_t)c * ld + k;
    float e0[4], e1[4], e2[4], wc[5], o[4];
    ld4(e0, ekin_e + (size_t)ce[0] * ld + k);
    ld4(e1, ekin_e + (size_t)ce[1] * ld + k);
    ld4(e2, ekin_e + (size_t)ce[2] * ld + k);
    {
      float a[4];
      ld4(a, w + i);
#pragma unroll
      for (int j = 0; j < 4; ++j) wc[j] = a[j];
      wc[4] = k + 4 <= nlev ? w[i + 4] : 0.0f;
    }
    const float q0 = q[0], q1 = q[1], q2 = q[2];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float s = q0 * e0[j];
      s += q1 * e1[j];
      s += q2 * e2[j];
      o[j] = s;
    }
    st4(ekin_c + i, o);
    if (wcc) {
      float a[4];
      ld4(a, wcc + i);
      const float b = k + 4 <= nlev ? wcc[i + 4] : 0.0f;
#pragma unroll
      for (int j = 0; j < 4; ++j) o[j] = (wc[j] - a[j]) + (wc[j + 1] - (j < 3 ? a[j < 3 ? j + 1 : 3] : b));
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) o[j] = wc[j] + wc[j + 1];
    }
    st4(wq + i, o);
    if (divd2) {
      const int* cc = g.c2e2c + 3 * (size_t)c;
      const float* L = g.lap_c + 3 * (size_t)c;
      float dc[4], d0[4], d1[4], d2[4];
      ld4(dc, divd + i);
      ld4(d0, divd + (size_t)cc[0] * ld + k);
      ld4(d1, divd + (size_t)cc[1] * ld + k);
      ld4(d2, divd + (size_t)cc[2] * ld + k);
      const float L0 = L[0], L1 = L[1], L2 = L[2];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float r = L0 * (d0[j] - dc[j]);
        r += L1 * (d1[j] - dc[j]);
        r += L2 * (d2[j] - dc[j]);
        o[j] = r;
      }
      st4(divd2 + i, o);
    }
    return;
  }
  t -= ncell;
  if (t >= (unsigned)g.nv * nqh) return;
  const int vx = (int)(t / (unsigned)nqh), k = 4 * (int)(t - (unsigned)vx * nqh);
  const int* ve = g.v2e + 6 * (size_t)vx;
  const int* vc = g.v2c + 6 * (size_t)vx;
  const float* cw = g.curl_v + 6 * (size_t)vx;
  const float* rw = g.c2v_w + 6 * (size_t)vx;
  const size_t i = (size_t)vx * ld + k;
  if (k < nlev) {
    float z[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int m = 0; m < 6; ++m) {
      float x[4];
      ld4(x, vn + (size_t)ve[m] * ld + k);
      const float cm = cw[m];
#pragma unroll
      for (int j = 0; j < 4; ++j) z[j] += cm * x[j];
    }
    st4(zeta + i, z);
  }
  float s[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
  for (int m = 0; m < 6; ++m) {
    float x[4];
    ld4(x, w + (size_t)vc[m] * ld + k);
    const float rm = rw[m];
#pragma unroll
    for (int j = 0; j < 4; ++j) s[j] += rm * x[j];
  }
  st4(w_v + i, s);
}

// A3, as va_edge_tend
template <bool kTerr>
__global__ void va_edge_tend_q(GridT<float> g, VertT<float> v, const float* __restrict__ vn_ie,
                               const float* __restrict__ w, const float* __restrict__ vt,
                               const float* __restrict__ ekin_c, const float* __restrict__ zeta,
                               const float* __restrict__ w_v, float* __restrict__ ddt_vn, float* __restrict__ gw_e,
                               TerrT<float> tr, const float* __restrict__ wq) {
  int e, k;
  const int nlev = v.nlev, ld = v.ldf;
  if (!quad_index(g.ne, quads_half(nlev), e, k)) return;
  const int2 cc = *reinterpret_cast<const int2*>(g.e2c + 2 * (size_t)e);
  const int2 vv = *reinterpret_cast<const int2*>(g.e2v + 2 * (size_t)e);
  const size_t i = (size_t)e * ld + k, i0 = (size_t)cc.x * ld + k, i1 = (size_t)cc.y * ld + k;
  const size_t im = (size_t)vv.x * ld + k, ip = (size_t)vv.y * ld + k;
  float ie[5], te[5];  // vn at the half levels k .. k+4; vt at the levels k-1 .. k+3
  {
    float a[4];
    ld4(a, vn_ie + i);
#pragma unroll
    for (int j = 0; j < 4; ++j) ie[j] = a[j];
    ie[4] = k + 4 <= nlev ? vn_ie[i + 4] : 0.0f;
    ld4(a, vt + i);
#pragma unroll
    for (int j = 0; j < 4; ++j) te[j + 1] = a[j];
    te[0] = k > 0 ? vt[i - 1] : 0.0f;
  }
  if (k < nlev) {
    float q0[4], q1[4], zm[4], zp[4], k0[4], k1[4], qd[4], o[4];
    ld4(q0, wq + i0);
    ld4(q1, wq + i1);
    ld4(zm, zeta + im);
    ld4(zp, zeta + ip);
    ld4(k0, ekin_c + i0);
    ld4(k1, ekin_c + i1);
    ld4(qd, kTerr ? tr.qdz_e + i : v.qdz + k);
    const float fe = g.f_e[e], hd = g.hinv_d[e];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float ws = q0[j] + q1[j];
      const float adv = (ws * (ie[j] - ie[j + 1])) * qd[j];
      const float zf = fmat(0.5f, zm[j] + zp[j], fe);
      const float dk = k0[j] - k1[j];
      o[j] = fmat(dk, hd, fmat(zf, te[j + 1], -adv));
    }
    st4(ddt_vn + i, o);
  }
  float w0[4], w1[4], vm[4], vp[4], wg[4], o[4];
  ld4(w0, w + i0);
  ld4(w1, w + i1);
  ld4(vm, w_v + im);
  ld4(vp, w_v + ip);
  ld4(wg, kTerr ? tr.wgt_e + i : v.wgt + k);
  const float dol = g.d_o_l[e];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float gw = 0.0f;
    if (k + j > 0 && k + j < nlev) {
      const float vtie = te[j + 1] + wg[j] * (te[j] - te[j + 1]);
      const float dwn = w1[j] - w0[j];
      const float dwt = (vp[j] - vm[j]) * dol;
      gw = fmat(ie[j], dwn, vtie * dwt);
    }
    o[j] = gw;
  }
  st4(gw_e + i, o);
}

// A4, as va_cell_w
template <bool kTerr>
__global__ void va_cell_w_q(GridT<float> g, VertT<float> v, const float* __restrict__ w,
                            const float* __restrict__ gw_e, float* __restrict__ ddt_w, TerrT<float> tr,
                            const float* __restrict__ wcc) {
  int c, k;
  const int nlev = v.nlev, ld = v.ldf;
  if (!quad_index(g.nc, quads_half(nlev), c, k)) return;
  const int* ce = g.c2e + 3 * (size_t)c;
  const float* q = g.e2c_wd + 3 * (size_t)c;
  const size_t i = (size_t)c * ld + k;
  float g0[4], g1[4], g2[4], a[4], qd[4], cr[4], o[4], wc[6];  // w at the half levels k-1 .. k+4
  ld4(g0, gw_e + (size_t)ce[0] * ld + k);
  ld4(g1, gw_e + (size_t)ce[1] * ld + k);
  ld4(g2, gw_e + (size_t)ce[2] * ld + k);
  ld4(a, w + i);
#pragma unroll
  for (int j = 0; j < 4; ++j) wc[j + 1] = a[j];
  wc[0] = k > 0 ? w[i - 1] : 0.0f;
  wc[5] = k + 4 <= nlev ? w[i + 4] : 0.0f;
  ld4(qd, kTerr ? tr.qdzh_c + i : v.qdzh + k);
  if constexpr (kTerr) ld4(cr, wcc + i);
  const float q0 = q[0], q1 = q[1], q2 = q[2];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float r = 0.0f;
    if (k + j > 0 && k + j < nlev) {
      const float h = fmat(q2, g2[j], fmat(q1, g1[j], q0 * g0[j]));
      const float wa = kTerr ? wc[j + 1] - cr[j] : wc[j + 1];
      r = fmat(-(wa * (wc[j] - wc[j + 2])), qd[j], -h);
    }
    o[j] = r;
  }
  st4(ddt_w + i, o);
}

// A5, as sn_cell_grad; pairs: rows of nlev FP64 values may be read two at a
// time (an even nlev and 16-byte aligned arrays)
template <bool kTerr>
__global__ void sn_cell_grad_q(GridT<float> g, VertT<float> v, const float* __restrict__ rho,
                               const float* __restrict__ theta, float* __restrict__ grad4,
                               const double* __restrict__ exner, const double* __restrict__ exner_pr, double exfac,
                               df* __restrict__ pex, const double* __restrict__ exner_ref_c, bool pairs) {
  int c, k;
  const int nlev = v.nlev, ld = v.ldf;
  if (!quad_index(g.nc, quads_full(nlev), c, k)) return;
  const size_t n = (size_t)g.nc * ld;
  const int* cc = g.c2e2c + 3 * (size_t)c;
  const float* G = g.grad_c + 6 * (size_t)c;
  const size_t i = (size_t)c * ld + k, is = (size_t)c * nlev + k;
  double ex[4], pr[4];
  if (pairs) {
#pragma unroll
    for (int j = 0; j < 4; j += 2)
      if (k + j < nlev) {
        const double2 a = *reinterpret_cast<const double2*>(exner + is + j);
        const double2 b = *reinterpret_cast<const double2*>(exner_pr + is + j);
        ex[j] = a.x, ex[j + 1] = a.y, pr[j] = b.x, pr[j + 1] = b.y;
      }
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (k + j < nlev) ex[j] = exner[is + j], pr[j] = exner_pr[is + j];
  }
  float r[4], r0[4], r1[4], r2[4], t[4], t0[4], t1[4], t2[4], o[4];
  const size_t i0 = (size_t)cc[0] * ld + k, i1 = (size_t)cc[1] * ld + k, i2 = (size_t)cc[2] * ld + k;
  ld4(r, rho + i);
  ld4(r0, rho + i0);
  ld4(r1, rho + i1);
  ld4(r2, rho + i2);
  ld4(t, theta + i);
  ld4(t0, theta + i0);
  ld4(t1, theta + i1);
  ld4(t2, theta + i2);
  // extrapolated exner perturbation (1 + a) pr - a pr_old as a double-word pair
  // (exner is near 1, the difference across an edge ~1e-5 of it)
  const df a = to_df(1.0 + exfac), b = to_df(exfac);
  df p[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    p[j] = {0.0f, 0.0f};
    if (k + j < nlev) {
      const double ex_ref = kTerr ? exner_ref_c[is + j] : v.exner_ref[k + j];
      p[j] = a * (to_df(ex[j]) - to_df(ex_ref)) - b * to_df(pr[j]);
    }
  }
  st4(pex + i, p);
  const float G0 = G[0], G1 = G[1], G2 = G[2], G3 = G[3], G4 = G[4], G5 = G[5];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    r0[j] = r0[j] - r[j], r1[j] = r1[j] - r[j], r2[j] = r2[j] - r[j];
    t0[j] = t0[j] - t[j], t1[j] = t1[j] - t[j], t2[j] = t2[j] - t[j];
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) o[j] = G0 * r0[j] + G2 * r1[j] + G4 * r2[j];
  st4(grad4 + i, o);
#pragma unroll
  for (int j = 0; j < 4; ++j) o[j] = G1 * r0[j] + G3 * r1[j] + G5 * r2[j];
  st4(grad4 + n + i, o);
#pragma unroll
  for (int j = 0; j < 4; ++j) o[j] = G0 * t0[j] + G2 * t1[j] + G4 * t2[j];
  st4(grad4 + 2 * n + i, o);
#pragma unroll
  for (int j = 0; j < 4; ++j) o[j] = G1 * t0[j] + G3 * t1[j] + G5 * t2[j];
  st4(grad4 + 3 * n + i, o);
}

// A6, as sn_edge_pred, from the perturbations of rho and theta_v, with the
// reference added back; the difference of the exner perturbations across the
// edge is taken of double-word pairs (neighbours agree to 4-5 digits, more than
// FP32 carries).  A quad's levels mostly share their upwind cell: its fields come
// as quads then, else level by level.
template <bool kTerr>
__global__ void sn_edge_pred_q(GridT<float> g, VertT<float> v, ScalT<float> sc, const float* __restrict__ vn,
                               const float* __restrict__ vt, const float* __restrict__ ddt_vn,
                               const float* __restrict__ rho, const float* __restrict__ theta,
                               const df* __restrict__ pex, const float* __restrict__ grad4, float* __restrict__ rho_e,
                               float* __restrict__ theta_e, float* __restrict__ hpg, float* __restrict__ vn_p,
                               TerrT<float> tr) {
  int e, k;
  const int nlev = v.nlev, ld = v.ldf;
  if (!quad_index(g.ne, quads_full(nlev), e, k)) return;
  const size_t n = (size_t)g.nc * ld;
  const int2 cc = *reinterpret_cast<const int2*>(g.e2c + 2 * (size_t)e);
  const size_t i = (size_t)e * ld + k, i0 = (size_t)cc.x * ld + k, i1 = (size_t)cc.y * ld + k;
  float x[4], t[4], dd[4];
  df p0[4], p1[4];
  ld4(x, vn + i);
  ld4(p0, pex + i0);
  ld4(p1, pex + i1);
  ld4(t, vt + i);
  ld4(dd, ddt_vn + i);
  bool up[4];  // upwind from the edge's second cell
#pragma unroll
  for (int j = 0; j < 4; ++j) up[j] = !(x[j] >= 0.0f);
#pragma unroll
  for (int j = 1; j < 4; ++j)
    if (k + j >= nlev) up[j] = up[0];  // pads: no level of their own
  float ru[4], tu[4], ga[4], gb[4], gc[4], gd[4];
  if (up[0] == up[1] && up[0] == up[2] && up[0] == up[3]) {
    const size_t iu = up[0] ? i1 : i0;
    ld4(ru, rho + iu);
    ld4(tu, theta + iu);
    ld4(ga, grad4 + iu);
    ld4(gb, grad4 + n + iu);
    ld4(gc, grad4 + 2 * n + iu);
    ld4(gd, grad4 + 3 * n + iu);
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const size_t iu = (up[j] ? i1 : i0) + j;
      ru[j] = rho[iu];
      tu[j] = theta[iu];
      ga[j] = grad4[iu];
      gb[j] = grad4[n + iu];
      gc[j] = grad4[2 * n + iu];
      gd[j] = grad4[3 * n + iu];
    }
  }
  float rr[4], tref[4];
  ld4(rr, v.rho_ref + k);
  ld4(tref, v.theta_ref + k);
  // the two cells' offsets of the back trajectory
  float u[12];
  {
    const float4* up4 = reinterpret_cast<const float4*>(g.upw_s + 12 * (size_t)e);
    const float4 a = up4[0], b = up4[1], c = up4[2];
    u[0] = a.x, u[1] = a.y, u[2] = a.z, u[3] = a.w, u[4] = b.x, u[5] = b.y;
    u[6] = b.z, u[7] = b.w, u[8] = c.x, u[9] = c.y, u[10] = c.z, u[11] = c.w;
  }
  const float cid = g.cpd_inv_d[e];
  // over terrain: the pairs above and below the quad, the vertical spacings and the slope
  [[maybe_unused]] df pm0{0.f, 0.f}, pm1{0.f, 0.f}, pn0{0.f, 0.f}, pn1{0.f, 0.f};
  [[maybe_unused]] float idz0[4], idz1[4], sl[4];
  if constexpr (kTerr) {
    if (k > 0) pm0 = pex[i0 - 1], pm1 = pex[i1 - 1];
    if (k + 4 < nlev) pn0 = pex[i0 + 4], pn1 = pex[i1 + 4];
    ld4(idz0, tr.inv_dzm_c + i0);
    ld4(idz1, tr.inv_dzm_c + i1);
    ld4(sl, tr.ddxn_mc + i);
  }
  float o_r[4], o_t[4], o_h[4], o_v[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float vne = x[j], vte = t[j];
    const float ax = up[j] ? u[6] : u[0], ay = up[j] ? u[7] : u[1], nx = up[j] ? u[8] : u[2],
                ny = up[j] ? u[9] : u[3], tx = up[j] ? u[10] : u[4], ty = up[j] ? u[11] : u[5];
    const float dx = fmat(-vne, nx, fmat(-vte, tx, ax));
    const float dy = fmat(-vne, ny, fmat(-vte, ty, ay));
    const float rv = ru[j] + rr[j], tv = tu[j] + tref[j];
    const float re = fmat(ga[j], dx, fmat(gb[j], dy, rv));
    const float te = fmat(gc[j], dx, fmat(gd[j], dy, tv));
    float h;
    if constexpr (kTerr) {
      h = 0.0f;
      const int kl = k + j;
      if (kl < nlev) {  // centred vertical differences, one-sided at the ends
        const df a0 = kl == 0 ? p0[0] : j == 0 ? pm0 : p0[j > 0 ? j - 1 : 0];
        const df a1 = kl == 0 ? p1[0] : j == 0 ? pm1 : p1[j > 0 ? j - 1 : 0];
        const df b0 = kl + 1 == nlev ? p0[j] : j == 3 ? pn0 : p0[j < 3 ? j + 1 : 3];
        const df b1 = kl + 1 == nlev ? p1[j] : j == 3 ? pn1 : p1[j < 3 ? j + 1 : 3];
        const float dz0 = to_float(a0 - b0) * idz0[j];
        const float dz1 = to_float(a1 - b1) * idz1[j];
        h = te * (to_float(p1[j] - p0[j]) * cid - sl[j] * (0.5f * (dz0 + dz1)));
      }
    } else {
      h = te * (to_float(p1[j] - p0[j]) * cid);
    }
    o_r[j] = re;
    o_t[j] = te;
    o_h[j] = h;
    o_v[j] = vne + sc.dt_s * (dd[j] - h);
  }
  st4(rho_e + i, o_r);
  st4(theta_e + i, o_t);
  st4(hpg + i, o_h);
  st4(vn_p + i, o_v);
}

// the cell divergence, as sn_cell_div (pairs: as in sn_cell_grad_q)
template <bool kTerr>
__global__ void sn_cell_div_q(GridT<float> g, VertT<float> v, const float* __restrict__ vn, float* __restrict__ divd,
                              const double* __restrict__ exner, double* __restrict__ exner_pr,
                              const double* __restrict__ exner_ref_c, bool pairs) {
  int c, k;
  const int nlev = v.nlev, ld = v.ldf;
  if (!quad_index(g.nc, quads_full(nlev), c, k)) return;
  const int* ce = g.c2e + 3 * (size_t)c;
  const float* dv = g.div_c + 3 * (size_t)c;
  float x0[4], x1[4], x2[4], o[4];
  ld4(x0, vn + (size_t)ce[0] * ld + k);
  ld4(x1, vn + (size_t)ce[1] * ld + k);
  ld4(x2, vn + (size_t)ce[2] * ld + k);
  const float d0 = dv[0], d1 = dv[1], d2 = dv[2];
#pragma unroll
  for (int j = 0; j < 4; ++j) o[j] = fmat(d2, x2[j], fmat(d1, x1[j], d0 * x0[j]));
  st4(divd + (size_t)c * ld + k, o);
  if (!exner_pr) return;
  const size_t is = (size_t)c * nlev + k;
  if (pairs) {
#pragma unroll
    for (int j = 0; j < 4; j += 2)
      if (k + j < nlev) {
        const double2 a = *reinterpret_cast<const double2*>(exner + is + j);
        const double2 b = *reinterpret_cast<const double2*>((kTerr ? exner_ref_c + is : v.exner_ref + k) + j);
        *reinterpret_cast<double2*>(exner_pr + is + j) = make_double2(a.x - b.x, a.y - b.y);
      }
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (k + j < nlev) exner_pr[is + j] = exner[is + j] - (kTerr ? exner_ref_c[is + j] : v.exner_ref[k + j]);
  }
}

// Divergences of the horizontal mass and theta fluxes, FP32 fluxes summed in
// double-word FP32 (mass conserved to about 2^-48 of the flux, without the
// slow FP64 pipe) and stored as the pair for the column solve:
//   vf_e = vn_e + divflux (D_c1 - D_c0)/d_e,  F_e = rho_e vf_e,
//   div_m = sum s l F / A,  div_t = sum s l F theta_e / A
// Over terrain (kTerr) each flux carries its edge layer thickness over the
// cell's, fx_ratio = dz_e / dz_c.  With an even nlev two levels' results are one
// aligned store.
template <bool kTerr>
__global__ void sn_cell_fluxdiv_q(GridT<float> g, VertT<float> v, const float* __restrict__ vn,
                                  const float* __restrict__ divd, const float* __restrict__ rho_e,
                                  const float* __restrict__ theta_e, df* __restrict__ div_m, df* __restrict__ div_t,
                                  const float* __restrict__ fx_ratio) {
  int c, k;
  const int nlev = v.nlev, ld = v.ldf;
  if (!quad_index(g.nc, quads_full(nlev), c, k)) return;
  const int* ce = g.c2e + 3 * (size_t)c;
  const df* dvp = reinterpret_cast<const df*>(g.div_c_hl) + 3 * (size_t)c;
  df dm[4] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}}, dt[4] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    const int e = ce[m];
    const int2 cc = *reinterpret_cast<const int2*>(g.e2c + 2 * (size_t)e);
    const size_t i = (size_t)e * ld + k;
    float x[4], d0[4], d1[4], r[4], th[4], fx[4];
    ld4(x, vn + i);
    ld4(d1, divd + (size_t)cc.y * ld + k);
    ld4(d0, divd + (size_t)cc.x * ld + k);
    ld4(r, rho_e + i);
    ld4(th, theta_e + i);
    if constexpr (kTerr) ld4(fx, fx_ratio + ((size_t)c * 3 + m) * ld + k);
    const float fd = g.fdiv_e[e];
    const df w = dvp[m];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float vf = x[j] + fd * (d1[j] - d0[j]);
      float f = r[j] * vf;
      if constexpr (kTerr) f = f * fx[j];
      const float ft = f * th[j];
      dm[j] = dm[j] + w * f;
      dt[j] = dt[j] + w * ft;
    }
  }
  const size_t is = (size_t)c * nlev + k;
  if ((nlev & 1) == 0) {
#pragma unroll
    for (int j = 0; j < 4; j += 2)
      if (k + j < nlev) {
        *reinterpret_cast<float4*>(div_m + is + j) = make_float4(dm[j].hi, dm[j].lo, dm[j + 1].hi, dm[j + 1].lo);
        *reinterpret_cast<float4*>(div_t + is + j) = make_float4(dt[j].hi, dt[j].lo, dt[j + 1].hi, dt[j + 1].lo);
      }
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (k + j < nlev) div_m[is + j] = dm[j], div_t[is + j] = dt[j];
  }
}

// A1-A2 over terrain, as va_concorr
__global__ void va_concorr_q(GridT<float> g, VertT<float> v, TerrT<float> tr, const float* __restrict__ vn_ie,
                             const float* __restrict__ vt, float* __restrict__ wcc) {
  int c, k;
  const int nlev = v.nlev, ld = v.ldf;
  if (!quad_index(g.nc, quads_half(nlev), c, k)) return;
  const int* ce = g.c2e + 3 * (size_t)c;
  const float* q = g.e2c_w + 3 * (size_t)c;
  float s[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    const size_t i = (size_t)ce[m] * ld + k;
    float a[4], y[4], wg[4], sn[4], st[4];
    ld4(a, vn_ie + i);
    ld4(y, vt + i);
    ld4(wg, tr.wgt_e + i);
    ld4(sn, tr.ddxn_ifc + i);
    ld4(st, tr.ddxt_ifc + i);
    const float ym = k > 0 ? vt[i - 1] : 0.0f, qm = q[m];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float up = j == 0 ? ym : y[j > 0 ? j - 1 : 0];
      const float b = k + j == nlev ? up : y[j] + wg[j] * (up - y[j]);
      if (k + j > 0) s[j] += qm * (a[j] * sn[j] + b * st[j]);
    }
  }
  st4(wcc + (size_t)c * ld + k, s);
}

// four consecutive FP64 values of a row of n from level k on (in pairs where
// the row allows it), and their store
__device__ __forceinline__ void ld4(double (&a)[4], const double* p, int k, int n, bool pairs) {
#pragma unroll
  for (int j = 0; j < 4; j += 2) {
    if (pairs) {
      if (k + j < n) {
        const double2 x = *reinterpret_cast<const double2*>(p + j);
        a[j] = x.x, a[j + 1] = x.y;
      }
    } else {
      if (k + j < n) a[j] = p[j];
      if (k + j + 1 < n) a[j + 1] = p[j + 1];
    }
  }
}
__device__ __forceinline__ void st4(double* p, const double (&a)[4], int k, int n, bool pairs) {
#pragma unroll
  for (int j = 0; j < 4; j += 2) {
    if (pairs) {
      if (k + j < n) *reinterpret_cast<double2*>(p + j) = make_double2(a[j], a[j + 1]);
    } else {
      if (k + j < n) p[j] = a[j];
      if (k + j + 1 < n) p[j + 1] = a[j + 1];
    }
  }
}

// Mixed mode: FP32 mirrors of the FP64 state at the start of a call (the
// caller may have changed the state between calls): the edges' full-level
// quads, then the cells' half-level quads.
__global__ void mx_refresh(int ne, int nc, VertT<float> v, const double* __restrict__ theta_ref,
                           const double* __restrict__ rho_ref, StateView st, Mirrors m, bool pairs) {
  const int nlev = v.nlev, ld = v.ldf, nqf = quads_full(nlev), nqh = quads_half(nlev);
  unsigned t = flat_thread();
  const unsigned nedge = (unsigned)ne * nqf;
  double x[4] = {}, y[4] = {};
  float o[4];
  if (t < nedge) {
    const int e = (int)(t / (unsigned)nqf), k = 4 * (int)(t - (unsigned)e * nqf);
    ld4(x, st.vn + (size_t)e * nlev + k, k, nlev, pairs);
#pragma unroll
    for (int j = 0; j < 4; ++j) o[j] = d2f(x[j]);
    st4(m.vn + (size_t)e * ld + k, o);
    return;
  }
  t -= nedge;
  if (t >= (unsigned)nc * nqh) return;
  const int c = (int)(t / (unsigned)nqh), k = 4 * (int)(t - (unsigned)c * nqh);
  const size_t q = (size_t)c * ld + k, is = (size_t)c * nlev + k;
  ld4(x, st.w + (size_t)c * (nlev + 1) + k, k, nlev + 1, false);
#pragma unroll
  for (int j = 0; j < 4; ++j) o[j] = d2f(x[j]);
  st4(m.w + q, o);
  if (k >= nlev) return;
  ld4(x, st.rho + is, k, nlev, pairs);
  ld4(y, st.theta_v + is, k, nlev, pairs);
#pragma unroll
  for (int j = 0; j < 4; ++j) o[j] = k + j < nlev ? d2f(x[j] - rho_ref[k + j]) : 0.0f;
  st4(m.rho + q, o);
#pragma unroll
  for (int j = 0; j < 4; ++j) o[j] = k + j < nlev ? d2f(y[j] - theta_ref[k + j]) : 0.0f;
  st4(m.th + q, o);
}

// A10, as diff_div_curl_uv
__global__ void diff_div_curl_uv_q(GridT<float> g, VertT<float> v, const float* __restrict__ vn,
                                   float* __restrict__ div_vn, float* __restrict__ zeta, float* __restrict__ uv3) {
  const int nlev = v.nlev, ld = v.ldf, nq = quads_full(nlev);
  unsigned t = flat_thread();
  const unsigned ncell = (unsigned)g.nc * nq;
  if (t < ncell) {
    const int c = (int)(t / (unsigned)nq), k = 4 * (int)(t - (unsigned)c * nq);
    const int* ce = g.c2e + 3 * (size_t)c;
    const float* dv = g.div_c + 3 * (size_t)c;
    float x0[4], x1[4], x2[4], o[4];
    ld4(x0, vn + (size_t)ce[0] * ld + k);
    ld4(x1, vn + (size_t)ce[1] * ld + k);
    ld4(x2, vn + (size_t)ce[2] * ld + k);
    const float d0 = dv[0], d1 = dv[1], d2 = dv[2];
#pragma unroll
    for (int j = 0; j < 4; ++j) o[j] = d0 * x0[j] + d1 * x1[j] + d2 * x2[j];
    st4(div_vn + (size_t)c * ld + k, o);
    return;
  }
  t -= ncell;
  if (t >= (unsigned)g.nv * nq) return;
  const int vx = (int)(t / (unsigned)nq), k = 4 * (int)(t - (unsigned)vx * nq);
  const size_t nvl = (size_t)g.nv * ld, i = (size_t)vx * ld + k;
  const int* ve = g.v2e + 6 * (size_t)vx;
  const float* cw = g.curl_v + 6 * (size_t)vx;
  const float* U = g.uv_w + 18 * (size_t)vx;
  float z[4] = {}, ux[4] = {}, uy[4] = {}, uz[4] = {};
#pragma unroll
  for (int m = 0; m < 6; ++m) {
    float x[4];
    ld4(x, vn + (size_t)ve[m] * ld + k);
    const float a = cw[m], b0 = U[3 * m], b1 = U[3 * m + 1], b2 = U[3 * m + 2];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      z[j] += a * x[j];
      ux[j] += b0 * x[j];
      uy[j] += b1 * x[j];
      uz[j] += b2 * x[j];
    }
  }
  st4(zeta + i, z);
  st4(uv3 + i, ux);
  st4(uv3 + nvl + i, uy);
  st4(uv3 + 2 * nvl + i, uz);
}

// a . b, the second product rounded by itself
__device__ __forceinline__ float dot3(float a0, float a1, float a2, float b0, float b1, float b2) {
  return fmaf(a2, b2, fmaf(a0, b0, a1 * b1));
}

// A10, as diff_edge_smag; which product of a sum is fused is written out here,
// since the compiler's choice depends on how it pairs the four levels
__global__ void diff_edge_smag_q(GridT<float> g, VertT<float> v, const float* __restrict__ div_vn,
                                 const float* __restrict__ zeta, const float* __restrict__ uv3,
                                 float* __restrict__ nu, float* __restrict__ lap) {
  int e, k;
  const int nlev = v.nlev, ld = v.ldf;
  if (!quad_index(g.ne, quads_full(nlev), e, k)) return;
  const size_t nvl = (size_t)g.nv * ld;
  const int4 dm = *reinterpret_cast<const int4*>(g.e2c2v + 4 * (size_t)e);
  const int2 cc = *reinterpret_cast<const int2*>(g.e2c + 2 * (size_t)e);
  const size_t im = (size_t)dm.x * ld + k, ip = (size_t)dm.y * ld + k;
  const size_t i2 = (size_t)dm.z * ld + k, i3 = (size_t)dm.w * ld + k;
  float dt[3][4], dn[3][4];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    float x[4], y[4];
    ld4(x, uv3 + a * nvl + ip);
    ld4(y, uv3 + a * nvl + im);
#pragma unroll
    for (int j = 0; j < 4; ++j) dt[a][j] = x[j] - y[j];
    ld4(x, uv3 + a * nvl + i3);
    ld4(y, uv3 + a * nvl + i2);
#pragma unroll
    for (int j = 0; j < 4; ++j) dn[a][j] = x[j] - y[j];
  }
  float zp[4], zm[4], d0[4], d1[4];
  ld4(zp, zeta + ip);
  ld4(zm, zeta + im);
  ld4(d0, div_vn + (size_t)cc.x * ld + k);
  ld4(d1, div_vn + (size_t)cc.y * ld + k);
  const float* nt = g.nt + 6 * (size_t)e;
  const float n0 = nt[0], n1 = nt[1], n2 = nt[2], t0 = nt[3], t1 = nt[4], t2 = nt[5];
  const float il = g.inv_l[e], idn = g.inv_dn[e], sa = g.smag_a[e], id = g.inv_d[e];
  float o_nu[4], o_lap[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float dnx = dn[0][j], dny = dn[1][j], dnz = dn[2][j], dtx = dt[0][j], dty = dt[1][j], dtz = dt[2][j];
    const float tension = fmaf(dot3(dnx, dny, dnz, n0, n1, n2), idn, -(dot3(dtx, dty, dtz, t0, t1, t2) * il));
    const float shear = fmaf(dot3(dtx, dty, dtz, n0, n1, n2), il, dot3(dnx, dny, dnz, t0, t1, t2) * idn);
    o_nu[j] = sa * sqrtf(fmaf(tension, tension, shear * shear));
    o_lap[j] = (d1[j] - d0[j]) * id - (zp[j] - zm[j]) * il;
  }
  const size_t i = (size_t)e * ld + k;
  st4(nu + i, o_nu);
  st4(lap + i, o_lap);
}

// A10, as diff_second: the cells' half-level quads, then the vertices'
// full-level quads
__global__ void diff_second_q(GridT<float> g, VertT<float> v, ScalT<float> sc, const float* __restrict__ lap,
                              const float* __restrict__ nu, const float* __restrict__ w,
                              const float* __restrict__ theta, float* __restrict__ div_l, float* __restrict__ lap_w,
                              float* __restrict__ dtheta, float* __restrict__ curl_l,
                              const float* __restrict__ tenh_ex) {
  const int nlev = v.nlev, ld = v.ldf, nqf = quads_full(nlev), nqh = quads_half(nlev);
  unsigned t = flat_thread();
  const unsigned ncell = (unsigned)g.nc * nqh;
  if (t < ncell) {
    const int c = (int)(t / (unsigned)nqh), k = 4 * (int)(t - (unsigned)c * nqh);
    const int* ce = g.c2e + 3 * (size_t)c;
    const int* cc = g.c2e2c + 3 * (size_t)c;
    const float* Lp = g.lap_c + 3 * (size_t)c;
    const float L0 = Lp[0], L1 = Lp[1], L2 = Lp[2];
    const int e0 = ce[0], e1 = ce[1], e2 = ce[2];
    const size_t i = (size_t)c * ld + k, i0 = (size_t)cc[0] * ld + k, i1 = (size_t)cc[1] * ld + k,
                 i2 = (size_t)cc[2] * ld + k;
    const size_t j0 = (size_t)e0 * ld + k, j1 = (size_t)e1 * ld + k, j2 = (size_t)e2 * ld + k;
    float x[4], x0[4], x1[4], x2[4], o[4];
    ld4(x, w + i);
    ld4(x0, w + i0);
    ld4(x1, w + i1);
    ld4(x2, w + i2);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float lw = L0 * (x0[j] - x[j]);
      lw += L1 * (x1[j] - x[j]);
      lw += L2 * (x2[j] - x[j]);
      o[j] = lw;
    }
    st4(lap_w + i, o);
    if (k >= nlev) return;
    const float* dv = g.div_c + 3 * (size_t)c;
    const float dv0 = dv[0], dv1 = dv[1], dv2 = dv[2];
    ld4(x0, lap + j0);
    ld4(x1, lap + j1);
    ld4(x2, lap + j2);
#pragma unroll
    for (int j = 0; j < 4; ++j) o[j] = dv0 * x0[j] + dv1 * x1[j] + dv2 * x2[j];
    st4(div_l + i, o);
    if (!sc.hdiff_temp) return;
    float n0[4], n1[4], n2[4];
    ld4(x, theta + i);
    ld4(x0, theta + i0);
    ld4(x1, theta + i1);
    ld4(x2, theta + i2);
    ld4(n0, nu + j0);
    ld4(n1, nu + j1);
    ld4(n2, nu + j2);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (k + j >= nlev - sc.tenh_levels && k + j < nlev) {
        // enhanced near-surface temperature diffusion: the edge coefficient
        // raised by fac A_e / dtime max(e_c, e_nbr)
        const float ex = tenh_ex[i + j];
        n0[j] += g.tenh_a[e0] * max(ex, tenh_ex[i0 + j]);
        n1[j] += g.tenh_a[e1] * max(ex, tenh_ex[i1 + j]);
        n2[j] += g.tenh_a[e2] * max(ex, tenh_ex[i2 + j]);
      }
      const float tc = x[j];
      float f = L0 * n0[j] * (x0[j] - tc);
      f += L1 * n1[j] * (x1[j] - tc);
      f += L2 * n2[j] * (x2[j] - tc);
      o[j] = sc.dtime * f;
    }
    st4(dtheta + i, o);
    return;
  }
  t -= ncell;
  if (t >= (unsigned)g.nv * nqf) return;
  const int vx = (int)(t / (unsigned)nqf), k = 4 * (int)(t - (unsigned)vx * nqf);
  const int* ve = g.v2e + 6 * (size_t)vx;
  const float* cw = g.curl_v + 6 * (size_t)vx;
  float z[4] = {};
#pragma unroll
  for (int m = 0; m < 6; ++m) {
    float x[4];
    ld4(x, lap + (size_t)ve[m] * ld + k);
    const float a = cw[m];
#pragma unroll
    for (int j = 0; j < 4; ++j) z[j] += a * x[j];
  }
  st4(curl_l + (size_t)vx * ld + k, z);
}

// A10, as diff_edge_update (pairs: the state's rows, as in sn_cell_grad_q)
__global__ void diff_edge_update_q(GridT<float> g, VertT<float> v, ScalT<float> sc, double* __restrict__ vn,
                                   const float* __restrict__ nu, const float* __restrict__ lap,
                                   const float* __restrict__ div_l, const float* __restrict__ curl_l,
                                   float* __restrict__ m_vn, bool pairs) {
  int e, k;
  const int nlev = v.nlev, ld = v.ldf;
  if (!quad_index(g.ne, quads_full(nlev), e, k)) return;
  const int2 cc = *reinterpret_cast<const int2*>(g.e2c + 2 * (size_t)e);
  const int2 vv = *reinterpret_cast<const int2*>(g.e2v + 2 * (size_t)e);
  const size_t i = (size_t)e * ld + k;
  double* pv = vn + (size_t)e * nlev + k;
  double x[4] = {};
  float n[4], l[4], d0[4], d1[4], cm[4], cp[4], o[4];
  ld4(x, pv, k, nlev, pairs);
  ld4(n, nu + i);
  ld4(l, lap + i);
  ld4(d0, div_l + (size_t)cc.x * ld + k);
  ld4(d1, div_l + (size_t)cc.y * ld + k);
  ld4(cm, curl_l + (size_t)vv.x * ld + k);
  ld4(cp, curl_l + (size_t)vv.y * ld + k);
  const float id = g.inv_d[e], il = g.inv_l[e], k4 = g.k4_a[e];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float lap2 = (d1[j] - d0[j]) * id - (cp[j] - cm[j]) * il;
    const float inc = sc.dtime * n[j] * l[j] - k4 * lap2;
    x[j] = x[j] + f2d(inc);
    o[j] = d2f(x[j]);
  }
  st4(pv, x, k, nlev, pairs);
  st4(m_vn + i, o);
}

// A10, as diff_cell_update (pairs: the state's full-level rows)
__global__ void diff_cell_update_q(GridT<float> g, VertT<float> v, ScalT<float> sc,
                                   const double* __restrict__ theta_ref, double rd_o_cvd, StateView st,
                                   const float* __restrict__ lap_w, const float* __restrict__ dtheta, Mirrors m,
                                   bool pairs) {
  int c, k;
  const int nlev = v.nlev, nlevp = nlev + 1, ld = v.ldf;
  if (!quad_index(g.nc, quads_half(nlev), c, k)) return;
  const int* cc = g.c2e2c + 3 * (size_t)c;
  const float* Lp = g.lap_c + 3 * (size_t)c;
  const float L0 = Lp[0], L1 = Lp[1], L2 = Lp[2], k4 = g.k4w_c[c];
  const size_t i = (size_t)c * ld + k;
  float x[4], x0[4], x1[4], x2[4], o[4];
  ld4(x, lap_w + i);
  ld4(x0, lap_w + (size_t)cc[0] * ld + k);
  ld4(x1, lap_w + (size_t)cc[1] * ld + k);
  ld4(x2, lap_w + (size_t)cc[2] * ld + k);
  ld4(o, m.w + i);
  double* pw = st.w + (size_t)c * nlevp + k;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (k + j == 0 || k + j >= nlev) continue;
    float l2 = L0 * (x0[j] - x[j]);
    l2 += L1 * (x1[j] - x[j]);
    l2 += L2 * (x2[j] - x[j]);
    const double wn = pw[j] - f2d(k4 * l2);
    pw[j] = wn;
    o[j] = d2f(wn);
  }
  st4(m.w + i, o);
  if (k >= nlev || !sc.hdiff_temp) return;
  const size_t is = (size_t)c * nlev + k;
  double th[4] = {1.0, 1.0, 1.0, 1.0}, ex[4] = {};
  float dth[4];
  ld4(th, st.theta_v + is, k, nlev, pairs);
  ld4(ex, st.exner + is, k, nlev, pairs);
  ld4(dth, dtheta + i);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    o[j] = 0.0f;
    if (k + j >= nlev) continue;
    // exner (1 + rd/cvd dtheta/theta): the FP32 increment of a value near 1
    const double thn = th[j] + f2d(dth[j]);
    ex[j] = ex[j] + f2d(d2f(ex[j]) * ((float)rd_o_cvd * dth[j] / d2f(th[j])));
    th[j] = thn;
    o[j] = d2f(thn - theta_ref[k + j]);
  }
  st4(st.theta_v + is, th, k, nlev, pairs);
  st4(st.exner + is, ex, k, nlev, pairs);
  st4(m.th + i, o);
}

}  // namespace
}  // namespace icon
