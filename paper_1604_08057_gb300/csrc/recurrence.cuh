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

}  // namespace ov
