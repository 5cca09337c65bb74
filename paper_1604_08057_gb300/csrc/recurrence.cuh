// Device helpers shared by the kernels of the two-sided Lanczos recurrence.
#pragma once
#include "kernels.h"

namespace ov {

// ---------------------------------------------------------------------------
// helpers for the recurrence scalars
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool finite_z(zd a) { return isfinite(a.re) && isfinite(a.im); }

__device__ __forceinline__ void flag_error(SrcScal& sc, int bit, int step) {
  if (sc.err == 0) sc.err_step = step;
  sc.err |= bit;
}

// Sum NV partial slots of this source (fixed block order); thread 0 gets the result.
template <int NV>
__device__ __forceinline__ void sum_partials(const zd* part, int nblk, zd (&out)[NV], zd* scratch) {
  zd v[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) v[i] = mk(0.0, 0.0);
  // each thread takes a contiguous range of blocks, so the order is fixed
  for (int b = threadIdx.x; b < nblk; b += blockDim.x) {
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = v[i] + ld_cg(part + i * nblk + b);
  }
  block_sum<NV>(v, scratch);
#pragma unroll
  for (int i = 0; i < NV; ++i) out[i] = v[i];
}

// omega = s^dag r, rr = r^dag r, ss = s^dag s  ->  delta_{j+1}, beta_{j+1} and the next scales
template <typename R>
__device__ void omega_finalize(const Lat<R>& L, int src, int j, zd om, double rr, double ss) {
  SrcScal& sc = L.sc[src];
  const double aom = sqrt(om.re * om.re + om.im * om.im);
  if (!finite_z(om) || !isfinite(rr) || !isfinite(ss)) {
    flag_error(sc, ERRB_NONFINITE, j + 1);
    return;
  }
  if (aom <= 1e-14 * sqrt(rr * ss)) {
    flag_error(sc, ERRB_BREAKDOWN, j + 1);
    return;
  }
  const double d = sqrt(aom);
  const zd bt = mk(om.re / d, om.im / d);
  L.beta[(int64_t)src * L.k + j + 1] = bt;
  L.delta[(int64_t)src * L.k + j + 1] = d;
  sc.sv = mk(1.0 / d, 0.0);
  sc.sw = zdiv(mk(1.0, 0.0), conj(bt));
}

// bb = ||r||^2, sr = s^dag r of the start: beta_0 and the scales of v_1, w_1
template <typename R>
__device__ void init_finalize(const Lat<R>& L, int src, double bb, zd sr) {
  SrcScal& sc = L.sc[src];
  sc.err = 0;
  sc.err_step = -1;
  const double b0 = sqrt(bb);
  sc.beta0 = b0;
  if (!(b0 > 0.0) || !isfinite(b0)) flag_error(sc, ERRB_NONFINITE, 0);
  sc.sv = mk(1.0 / b0, 0.0);
  // w_1 = s sw with w_1^dag v_1 = 1: sw = beta_0 / conj(s^dag r); s = r in plain mode
  sc.sw = L.block ? zdiv(mk(b0, 0.0), conj(sr)) : mk(1.0 / b0, 0.0);
  L.beta[(int64_t)src * L.k] = mk(0.0, 0.0);
  L.delta[(int64_t)src * L.k] = 0.0;
}

// A1 = v_{j+1}^dag Gv, A2 = w_{j+1}^dag Gw in s: the reverse step's coefficients
template <typename R>
__device__ void rev_dots_epilogue(const Lat<R>& L, const Rev<R>& B, int src, int j, const zd (&s)[2]) {
  SrcScal& sc = L.sc[src];
  const int64_t o = (int64_t)src * L.k + j + 1;
  const double d = L.delta[o];
  const zd bt = L.beta[o];
  const zd om = mk(bt.re * d, bt.im * d);
  const double aom = d * d;
  double g_d = B.gdT[o] + sc.carry_delta - s[0].re / d;
  zd g_b = B.gbT[o] + sc.carry_beta - zdiv(conj(s[1]), conj(bt));
  zd g_w = mk(g_b.re / d, g_b.im / d);
  g_d -= (om.re * g_b.re + om.im * g_b.im) / (d * d);      // Re(conj(om) g_b)
  const double f = g_d / (2.0 * d * aom);
  g_w = g_w + mk(f * om.re, f * om.im);
  sc.cr1 = mk(1.0 / d, 0.0);
  sc.cr2 = conj(bt) * g_w;
  sc.cs1 = zdiv(mk(1.0, 0.0), bt);
  sc.cs2 = mk(d * g_w.re, -d * g_w.im);
  if (!finite_z(sc.cr2) || !finite_z(sc.cs2)) flag_error(sc, ERRB_NONFINITE, j);
}

// D1 = v_j^dag g_r, D2 = w_j^dag g_s, D3 = v_{j-1}^dag g_r, D4 = w_{j-1}^dag g_s -> g_alpha, carries
template <typename R>
__device__ void alpha_epilogue(const Lat<R>& L, const Rev<R>& B, int src, int j, const zd (&s)[4]) {
  SrcScal& sc = L.sc[src];
  const int64_t o = (int64_t)src * L.k + j;
  sc.g_alpha = B.gaT[o] - s[0] - conj(s[1]);
  if (j > 0) {
    sc.carry_beta = -s[2];
    sc.carry_delta = -s[3].re;
  } else {
    sc.carry_beta = mk(0.0, 0.0);
    sc.carry_delta = 0.0;
  }
}

// ---------------------------------------------------------------------------
// The same scalars formed by one warp: the divisions and square roots that do not depend on
// one another run in different lanes (each takes some 0.5 us at the FP64 rate, and these
// chains end every step's kernels: 14.9 us per update at 4^4, of which 5 are its fields).
// Every lane passes the same arguments.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double lane_of(double v, int l) { return __shfl_sync(0xffffffffu, v, l); }

template <typename R>
__device__ __forceinline__ void omega_finalize_warp(const Lat<R>& L, int src, int j, zd om, double rr, double ss) {
  const int lane = threadIdx.x & 31;
  SrcScal& sc = L.sc[src];
  const double q = sqrt(lane == 0 ? om.re * om.re + om.im * om.im : rr * ss);
  const double aom = lane_of(q, 0), rs = lane_of(q, 1);
  if (!finite_z(om) || !isfinite(rr) || !isfinite(ss)) {
    if (lane == 0) flag_error(sc, ERRB_NONFINITE, j + 1);
    return;
  }
  if (aom <= 1e-14 * rs) {
    if (lane == 0) flag_error(sc, ERRB_BREAKDOWN, j + 1);
    return;
  }
  const double d = sqrt(aom);
  const double y = (lane == 0 ? om.re : lane == 1 ? om.im : 1.0) / d;
  const zd bt = mk(lane_of(y, 0), lane_of(y, 1));
  const double sv = lane_of(y, 2);
  const double w = (lane == 0 ? bt.re : bt.im) / (bt.re * bt.re + bt.im * bt.im);   // 1 / conj(beta)
  const zd sw = mk(lane_of(w, 0), lane_of(w, 1));
  if (lane == 0) {
    L.beta[(int64_t)src * L.k + j + 1] = bt;
    L.delta[(int64_t)src * L.k + j + 1] = d;
    sc.sv = mk(sv, 0.0);
    sc.sw = sw;
  }
}

}  // namespace ov
