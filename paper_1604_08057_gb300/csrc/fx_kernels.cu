// The FP64 operator in block fixed point (fx.cuh): layout conversion and ov_apply_H.  Two
// threads (spins sp and 2 + sp) share a site.
#include "fx.cuh"
#include "kernels.h"

namespace ov {

static inline unsigned nblocks(int64_t n, int bs) { return (unsigned)((n + bs - 1) / bs); }

// ---------------------------------------------------------------------------
// links in fixed point
// ---------------------------------------------------------------------------
// Direction d = blockIdx.y: the links (d < 3 spatial, 3: ef U_t, 4: efinv U_t) of the
// user's array u.  The products are formed with their FP64 rounding errors, so each entry
// carries the fixed-point error alone.
__global__ void __launch_bounds__(128) k_pack_links_fx(const double* __restrict__ u, double ef, double efinv,
                                                       int4* __restrict__ out, short* __restrict__ ex, int64_t V) {
  const int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (x >= V) return;
  const int d = blockIdx.y, nu = d < 3 ? d : 3;
  const double f = d < 3 ? 1.0 : (d == 3 ? ef : efinv);
  const double2* iu = reinterpret_cast<const double2*>(u) + x * 36 + nu * 9;
  double hi[18], lo[18];
  unsigned mag = 0u;
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    const double2 a = iu[q];
    hi[2 * q] = f * a.x;
    hi[2 * q + 1] = f * a.y;
    lo[2 * q] = d < 3 ? 0.0 : fma(f, a.x, -hi[2 * q]);
    lo[2 * q + 1] = d < 3 ? 0.0 : fma(f, a.y, -hi[2 * q + 1]);
    mag = max(mag, max(fx_mag(hi[2 * q]), fx_mag(hi[2 * q + 1])));
  }
  const int eb = (int)(mag >> 20);
  const bool bad = mag != 0u && (eb < FX_U_MIN || eb > FX_U_MAX);
  const int ee = mag == 0u ? FX_U_MIN : eb;   // (a zero link does not raise a sum's scale)
  ex[(int64_t)d * V + x] = (short)(bad ? FX_BAD : ee);
  // u 2^(1081 - e): 59 bits; the error terms are at most 2^-53 of the largest entry
  const double f2 = fx_pow2(1081 - (bad ? 1022 : ee));
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    FxInt r{0, 0}, i{0, 0};
    if (!bad) {
      r = fx_split(4 * fx_conv(hi[2 * q], ee) + __double2ll_rn(f2 * lo[2 * q]));
      i = fx_split(4 * fx_conv(hi[2 * q + 1], ee) + __double2ll_rn(f2 * lo[2 * q + 1]));
    }
    out[fx_link_at(x, d) + q * 32] = make_int4(r.h, r.l, i.h, i.l);
  }
}
void pack_links_fx(const double* u, int4* out, short* ex, int64_t V, double ef, double efinv, cudaStream_t st) {
  k_pack_links_fx<<<dim3(nblocks(V, 128), 5), 128, 0, st>>>(u, ef, efinv, out, ex, V);
}

// ---------------------------------------------------------------------------
// user fields [src][site][12] (complex128).  A warp's 16 sites are 3 KB in a row there:
// both directions go through shared memory, so that global accesses are contiguous.
// ---------------------------------------------------------------------------
constexpr int kStage = 16 * 13;   // double2 per warp, rows padded by one
__device__ __forceinline__ void aos_load(const double* aos, int64_t src, int64_t V, int64_t x0, double2* st, int sp,
                                         zd (&p)[6]) {
  const int lane = threadIdx.x & 31;
  const int n = (int)min((int64_t)16, V - x0) * 12;
  const double2* in = reinterpret_cast<const double2*>(aos) + (src * V + x0) * 12;
  for (int i = lane; i < 192; i += 32) st[i / 12 * 13 + i % 12] = i < n ? in[i] : make_double2(0.0, 0.0);
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const double2 t = st[(lane & 15) * 13 + fx_comp(sp, i)];
    p[i] = mk(t.x, t.y);
  }
  __syncwarp();
}
__device__ __forceinline__ void aos_store(double* aos, int64_t src, int64_t V, int64_t x0, double2* st, int sp,
                                          const zd (&p)[6]) {
  const int lane = threadIdx.x & 31;
  const int n = (int)min((int64_t)16, V - x0) * 12;
#pragma unroll
  for (int i = 0; i < 6; ++i) st[(lane & 15) * 13 + fx_comp(sp, i)] = make_double2(p[i].re, p[i].im);
  __syncwarp();
  double2* o = reinterpret_cast<double2*>(aos) + (src * V + x0) * 12;
  for (int i = lane; i < n; i += 32) o[i] = st[i / 12 * 13 + i % 12];
  __syncwarp();
}
__device__ __forceinline__ void soa_store(double* f, int64_t V, int64_t s, int sp, const zd (&p)[6]) {
  double2* q = reinterpret_cast<double2*>(f) + s;
#pragma unroll
  for (int i = 0; i < 6; ++i) q[fx_comp(sp, i) * V] = make_double2(p[i].re, p[i].im);
}

// user spinors to fixed point; marked sites keep FP64 values in d, site-major
__global__ void __launch_bounds__(128) k_fx_pack(const double* __restrict__ aos, FxField f, double* __restrict__ d,
                                                 int64_t V, int64_t vs) {
  __shared__ double2 stage[4][kStage];
  const int sp = fx_spin_of(threadIdx.x), w = threadIdx.x >> 5;
  const int64_t x0 = blockIdx.x * (int64_t)64 + w * 16, x = x0 + (threadIdx.x & 15);
  const int src = blockIdx.y;
  if (x0 >= V) return;   // whole warps
  zd p[6];
  FxH o;
  aos_load(aos, src, V, x0, stage[w], sp, p);
  fx_from_double(p, o);
  if (x >= V) return;
  fx_put(fx_src(f, src, vs), x, sp, o);
  if (o.e == FX_BAD) soa_store(d + src * vs, V, x, sp, p);
}
void fx_pack(const double* aos, const FxField& f, double* d, int nsrc, int64_t V, int64_t vs, cudaStream_t st) {
  k_fx_pack<<<dim3(nblocks(V, 64), nsrc), 128, 0, st>>>(aos, f, d, V, vs);
}
// an FP64 site-major field to fixed point
__global__ void __launch_bounds__(128) k_fx_encode(const double* __restrict__ d, FxField f, int64_t V, int64_t vs) {
  const int sp = fx_spin_of(threadIdx.x);
  const int64_t x = blockIdx.x * (int64_t)64 + fx_site_of(threadIdx.x);
  const int src = blockIdx.y;
  const bool live = x < V;
  const double2* q = reinterpret_cast<const double2*>(d + src * vs);
  zd p[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const double2 t = live ? q[fx_comp(sp, i) * V + x] : make_double2(0.0, 0.0);
    p[i] = mk(t.x, t.y);
  }
  FxH o;
  fx_from_double(p, o);
  if (live) fx_put(fx_src(f, src, vs), x, sp, o);
}
void fx_encode(const double* d, const FxField& f, int nsrc, int64_t V, int64_t vs, cudaStream_t st) {
  k_fx_encode<<<dim3(nblocks(V, 64), nsrc), 128, 0, st>>>(d, f, V, vs);
}

// ---------------------------------------------------------------------------
// ov_apply_H
// ---------------------------------------------------------------------------
// FP64 hop sum from the user's links [site][direction][3][3] (out of line: reached only where
// a site or link is marked or the products may under- or overflow)
template <int NU>
__device__ __forceinline__ void hops_fp64_dir(Spinor<double>& acc, const FxLoad& ld, const double2* u, const Geom& g,
                                              int64_t x, const int c[4], double ff, double fb) {
  Spinor<double> nb;
  Half<double> h, uh;
  Mat3<double> m;
  ld(neighbour(g, x, c, NU, +1), nb);
  for (int e = 0; e < 9; ++e) m.m[e] = mk(u[x * 36 + NU * 9 + e].x, u[x * 36 + NU * 9 + e].y);
  spin_project<NU, +1>(nb, h);
  link_mul(m, h, uh);
  spin_reconstruct_add<NU, +1>(acc, uh, ff);
  const int64_t xb = neighbour(g, x, c, NU, -1);
  ld(xb, nb);
  for (int e = 0; e < 9; ++e) m.m[e] = mk(u[xb * 36 + NU * 9 + e].x, u[xb * 36 + NU * 9 + e].y);
  spin_project<NU, -1>(nb, h);
  link_dag_mul(m, h, uh);
  spin_reconstruct_add<NU, -1>(acc, uh, fb);
}
__device__ __noinline__ void hops_fp64(const FxLoad& ld, const double* u, const Geom& g, int64_t x, double ft,
                                       double fti, Spinor<double>* a) {
  int c[4];
  site_coords(g, x, c);
  const double2* u2 = reinterpret_cast<const double2*>(u);
  Spinor<double> t;
  spinor_zero(t);
  hops_fp64_dir<0>(t, ld, u2, g, x, c, 1.0, 1.0);
  hops_fp64_dir<1>(t, ld, u2, g, x, c, 1.0, 1.0);
  hops_fp64_dir<2>(t, ld, u2, g, x, c, 1.0, 1.0);
  hops_fp64_dir<3>(t, ld, u2, g, x, c, ft, fti);
  *a = t;
}
__device__ __forceinline__ void fx_pick(const Spinor<double>& t, int sp, zd (&p)[6]) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    p[i] = sp ? t.c[3 + i] : t.c[i];
    p[3 + i] = sp ? t.c[9 + i] : t.c[6 + i];
  }
}

// Bound by instruction issue at four blocks per SM (128 registers): 49% of the issue slots, the
// rest waits on fixed latencies and loads; DRAM 22%.  H^dagger on 16 sources at 6x18^3 takes 245
// us here, 864 with FP64 arithmetic, of which the FP64 units need 608.
// Blocks of blockDim.x / 2 sites x blockDim.y sources, whose sources share the link loads
// through L1.  psi's own term is read in FP64: from aos, the user's array, where the output has
// its layout too, else (aos null) from the site-major din.
__global__ void __launch_bounds__(128, 4) k_fx_apply(const __grid_constant__ Lat<double> L, FxField in,
                                                     const double* __restrict__ din, const double* __restrict__ aos,
                                                     double* __restrict__ out, int dagger) {
  __shared__ FxStage stage[4];
  FxStage& S = stage[(threadIdx.y * blockDim.x + threadIdx.x) >> 5];
  const int sp = fx_spin_of(threadIdx.x);
  const int64_t x0 = blockIdx.x * (int64_t)(blockDim.x >> 1) + (threadIdx.x >> 5) * 16;
  const int src = blockIdx.y * blockDim.y + threadIdx.y;
  const int64_t V = L.g.V;
  if (src >= L.nsrc || x0 >= V) return;   // whole warps
  const bool live = x0 + (threadIdx.x & 15) < V;
  const int64_t x = min(x0 + (threadIdx.x & 15), V - 1);
  const FxField f = fx_src(in, src, L.vs);
  const double* d = din + (int64_t)src * L.vs;
  const FxSite s(L.g, x);
  FxHalf acc;
  FxExps ex;
  fx_zero(acc, fx_range(ex, f, L.fu, L.g, s, dagger));
  const bool ok = fx_scale_ok(acc.E);
  if (!ok) acc.E = FX_E_BIAS;
  fx_hops(acc, f, L.fu, L.g, s, ex, dagger, sp, S);
  zd a[6];
  if (ok) {
    fx_double(acc, a);
  } else {
    Spinor<double> t;
    hops_fp64(FxLoad{f, d, V}, L.uaos, L.g, x, dagger ? L.efinv : L.ef, dagger ? L.ef : L.efinv, &t);
    fx_pick(t, sp, a);
  }
  zd p[6];
  __syncwarp();
  if (aos) {
    aos_load(aos, src, V, x0, S.out, sp, p);
  } else {
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      const double2 t = reinterpret_cast<const double2*>(d)[fx_comp(sp, i) * V + x];
      p[i] = mk(t.x, t.y);
    }
  }
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const zd q = mk(fma(-L.kappa, a[i].re, p[i].re), fma(-L.kappa, a[i].im, p[i].im));
    a[i] = i < 3 ? q : -q;
  }
  if (aos) aos_store(out, src, V, x0, S.out, sp, a);
  else if (live) soa_store(out + (int64_t)src * L.vs, V, x, sp, a);
}
void fx_apply_h(const Lat<double>& L, const FxField& in, const double* d, const double* aos, double* out, int dagger,
                cudaStream_t st, int variant) {
  // threads per block in x (two per site) and sources per block, or (variant 0) the rule below
  static const int shapes[FX_APPLY_SHAPES][2] = {{64, 1}, {32, 1}, {64, 2}, {32, 2}, {32, 4}, {128, 1}};
  int sx, sy;
  if (variant > 0) {
    const int* s = shapes[fx_apply_shape(variant) - 1];
    sx = s[0];
    sy = s[1];
  } else if (L.g.V * L.nsrc < 152 * 128) {
    sx = 32;
    sy = 1;
  } else {
    sy = L.nsrc >= 4 ? 4 : L.nsrc >= 2 ? 2 : 1;
    sx = 128 / sy;
  }
  k_fx_apply<<<dim3(nblocks(L.g.V, sx / 2), nblocks(L.nsrc, sy)), dim3(sx, sy), 0, st>>>(L, in, d, aos, out, dagger);
}

}  // namespace ov
