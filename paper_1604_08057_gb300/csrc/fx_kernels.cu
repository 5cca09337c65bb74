// FP64 calls in block fixed point (fx.cuh): layout conversion, ov_apply_H, and the two-sided
// Lanczos recurrence with its Gram-Schmidt projections where x alone is wanted (see LAT_* in
// ov_api.cu).  Every kernel reads and writes fixed-point fields; FP64 is left for the
// recurrence's scalars and for what goes back to the caller.
//
// Two threads (spins sp and 2 + sp) share a site unless a kernel says otherwise; blocks
// whose two halves treat the two sides of the recurrence (r and s) exchange through shared
// memory.  All reductions are deterministic.
#include <algorithm>
#include <atomic>

#include "fx.cuh"
#include "kernels.h"
#include "recurrence.cuh"

namespace ov {

static inline unsigned nblocks(int64_t n, int bs) { return (unsigned)((n + bs - 1) / bs); }

// Every rule on launch shapes looks at the lattice alone, so that a source's sums have the
// same order whatever sources run beside it.
//
// Blocks of the two-sided kernels cover 32 sites at a time, or 16 where 32 would leave SMs
// without a block; the elementwise ones take several such groups in turn, so that one wave
// (four blocks per SM) covers the lattice and a block's reduction serves all its groups.
static inline int two_sided_sites(const Lat<double>& L) { return L.g.V < 152 * 32 ? 16 : 32; }
static inline unsigned one_wave(const Lat<double>& L, int sites) {
  return std::min(nblocks(L.g.V, sites), 4u * 152u);
}
// Four warps per 16 sites and side (see k_fx_tsl) where one warp leaves most of an SM idle.
// In the Lanczos step the split sums are the unsplit ones bit for bit (alpha's partials are
// added by two warps in both), so its rule may count the sources (8^4 with four sources: 23 ms
// of stencils with the split, 12 without); the projection's sums over terms are not.
static inline bool fx_split_exact(const Lat<double>& L) { return L.g.V < 152 * 32 && L.g.V * L.nsrc < 152 * 64; }

// a launch with dynamic shared memory, whose limit is raised once per kernel and device
// (every caller sets the same value)
template <auto K, typename... A>
static void fx_launch(dim3 grid, int threads, size_t smem, cudaStream_t st, const A&... a) {
  static std::atomic<unsigned long long> done{0ull};
  int dev = 0;
  cudaGetDevice(&dev);
  const unsigned long long bit = 1ull << (dev & 63);
  if (!(done.load() & bit)) {
    cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
    done.fetch_or(bit);
  }
  K<<<grid, threads, smem, st>>>(a...);
}

// vector j of a basis
__device__ __forceinline__ FxField fx_bv(const Lat<double>& L, int src, int j) {
  const int64_t i = (int64_t)src * L.kcap + (j - L.jbase);
  return FxField{reinterpret_cast<int4*>(L.bv) + i * (L.vs / 2), L.bve + i * (L.vs / 24)};
}
__device__ __forceinline__ FxField fx_bw(const Lat<double>& L, int src, int j) {
  const int64_t i = (int64_t)src * L.kcap + (j - L.jbase);
  return FxField{reinterpret_cast<int4*>(L.bw) + i * (L.vs / 2), L.bwe + i * (L.vs / 24)};
}

// ---------------------------------------------------------------------------
// links in fixed point
// ---------------------------------------------------------------------------
// Direction d = blockIdx.y: the links (d < 3 spatial, 3: ef U_t, 4: efinv U_t) of the
// user's array u.  The products are formed with their FP64 rounding errors, so each entry
// carries the fixed-point error alone.  flush: a link below the window is encoded with the
// smallest exponent instead of marked (the callers that never use the links in FP64).
__global__ void __launch_bounds__(128) k_pack_links_fx(const double* __restrict__ u, double ef, double efinv,
                                                       int4* __restrict__ out, short* __restrict__ ex, int64_t V,
                                                       int flush) {
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
  const bool low = mag == 0u || (flush && eb < FX_U_MIN);
  const bool bad = !low && (eb < FX_U_MIN || eb > FX_U_MAX);
  const int ee = low ? FX_U_MIN : eb;   // (a zero link does not raise a sum's scale)
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
void pack_links_fx(const double* u, int4* out, short* ex, int64_t V, double ef, double efinv, bool flush,
                   cudaStream_t st) {
  k_pack_links_fx<<<dim3(nblocks(V, 128), 5), 128, 0, st>>>(u, ef, efinv, out, ex, V, flush ? 1 : 0);
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

// user spinors to fixed point, in f and (if set) g.  With d marked sites keep their FP64 values
// there; without it sites below the window are zero: nothing reads them in FP64
__global__ void __launch_bounds__(128) k_fx_pack(const double* __restrict__ aos, FxField f, FxField g,
                                                 double* __restrict__ d, int64_t V, int64_t vs) {
  __shared__ double2 stage[4][kStage];
  const int sp = fx_spin_of(threadIdx.x), w = threadIdx.x >> 5;
  const int64_t x0 = blockIdx.x * (int64_t)64 + w * 16, x = x0 + (threadIdx.x & 15);
  const int src = blockIdx.y;
  if (x0 >= V) return;   // whole warps
  const bool live = x < V;
  zd p[6];
  FxH o;
  aos_load(aos, src, V, x0, stage[w], sp, p);
  fx_from_double(p, o, !d);
  if (!live) return;
  fx_put(fx_src(f, src, vs), x, sp, o);
  if (g.c) fx_put(fx_src(g, src, vs), x, sp, o);
  if (d && o.e == FX_BAD) soa_store(d + src * vs, V, x, sp, p);
}
void fx_pack(const double* aos, const FxField& f, const FxField& g, double* d, int nsrc, int64_t V, int64_t vs,
             cudaStream_t st) {
  k_fx_pack<<<dim3(nblocks(V, 64), nsrc), 128, 0, st>>>(aos, f, g, d, V, vs);
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
// a site or link is marked)
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
  fx_zero(acc, fx_range(ex, f, 0, L.fu, L.g, s, dagger));
  const bool ok = acc.E < FX_BAD;
  if (!ok) acc.E = FX_E_BIAS;
  fx_hops(acc, f, 0, L.fu, L.g, s, ex, dagger, sp, S);
  zd a[6];
  if (ok) {
    fx_double(acc, false, a);
  } else {
    Spinor<double> t;
    hops_fp64(FxLoad{f, d, V, 0}, L.uaos, L.g, x, dagger ? L.efinv : L.ef, dagger ? L.ef : L.efinv, &t);
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
  // threads per block in x (two per site) and sources per block: variant v > 0 takes shape v
  // of this table (modulo its length), 0 the rule below
  static const int shapes[][2] = {{128, 1}, {64, 1}, {32, 1}, {64, 2}, {32, 2}, {32, 4}, {128, 1}};
  int sx, sy;
  if (variant > 0) {
    const int* s = shapes[variant % 7];
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

// ---------------------------------------------------------------------------
// forward recurrence
// ---------------------------------------------------------------------------
// start: beta_0 = ||r||, scales of v_1 and w_1 (see k_tsl_init)
__global__ void __launch_bounds__(128) k_fx_init(const __grid_constant__ Lat<double> L) {
  __shared__ FxSumBuf<2, 128> sum;
  __shared__ zd scratch[2 * 32];
  const int sp = fx_spin_of(threadIdx.x);
  const int64_t x = blockIdx.x * (int64_t)64 + fx_site_of(threadIdx.x);
  const int src = blockIdx.y;
  zd v[2] = {mk(0.0, 0.0), mk(0.0, 0.0)};
  if (x < L.g.V) {
    FxH r;
    fx_load(fx_src(L.fr, src, L.vs), x, sp, r);
    v[0] = mk(fx_norm2(r), 0.0);
  }
  zd* part = L.part + src * L.part_stride;
  fx_block_partials(v, sum, part, blockDim.x >> 5);
  if (arrive_last(L.cnt + src * 16 + 0, gridDim.x)) {
    zd s[2];
    fx_sum_partials<2>(part, gridDim.x, s, scratch, blockDim.x >> 5);
    if (threadIdx.x == 0) init_finalize(L, src, s[0].re, s[1]);
  }
}
void fx_tsl_init(const Lat<double>& L, cudaStream_t st) {
  k_fx_init<<<dim3(nblocks(L.g.V, 64), L.nsrc), 128, 0, st>>>(L);
}

// +-(f + c t) of a thread's components: the lower spins negated (gamma5)
__device__ __forceinline__ bool h_finish(FxHalf& o, const FxH& f, const FxCoef& c, const FxH& t) {
  fx_zero(o, 0);
  bool ok = fx_add(o, f);
  ok = fx_axpy(o, c, t) && ok;
#pragma unroll
  for (int i = 3; i < 6; ++i) o.v[i] = FxZ{-o.v[i].re, -o.v[i].im};
  return ok;
}
__device__ __forceinline__ void alpha_finish(const Lat<double>& L, int src, int j, const zd* part, zd* scratch, int nw) {
  if (arrive_last(L.cnt + src * 16 + 1, gridDim.x)) {
    zd s[1];
    fx_sum_partials<1>(part, gridDim.x, s, scratch, nw);
    if (threadIdx.x == 0) {
      SrcScal& sc = L.sc[src];
      if (!finite_z(s[0])) flag_error(sc, ERRB_NONFINITE, j);
      L.alpha[(int64_t)src * L.k + j] = s[0];
    }
  }
}

// Step j: v_j = sv r, w_j = sw s, p = H v_j, q = H^dag w_j, alpha_j = w_j^dag p.  A block of
// 4 SX threads covers SX (16 or 32) sites; its first half of warps forms v_j and p, the
// second half w_j and q of the same sites, so the links of both products come from L1 and
// a small lattice spreads over more warps.  w_j crosses to the first half through shared
// memory for the dot product.  H v_j = +-(v_j - kappa sv a) from the hop sum a of r.
// Bound by instruction issue and latency (some 5500 instructions per warp; its bytes take 10
// us at 14x14^3): 57 us there, 149 in FP64, whose products the FP64 units alone took 120 for.
//
// SPLIT: on a lattice with too few sites to fill the GPU a step's time is the latency of a
// thread's chain of hops (22 us at 4^4), so four warps share a side's 16 sites, one
// direction each, and add their sums through shared memory (14 us).
template <int SPLIT>
__global__ void __launch_bounds__(SPLIT ? 256 : 128, SPLIT ? 2 : 4)
    k_fx_tsl(const __grid_constant__ Lat<double> L, int j, int need_q) {
  extern __shared__ __align__(16) unsigned char fx_smem[];
  FxStage* stage = reinterpret_cast<FxStage*>(fx_smem);
  __shared__ FxSumBuf<1, SPLIT ? 256 : 128> sum;
  __shared__ FxCoef cs[2][2];   // [side]: scale, -kappa scale
  __shared__ zd scratch[32];
  const int half = blockDim.x >> 1, wid = threadIdx.x >> 5, nw = half >> 5;   // nw warps per side
  const bool left = threadIdx.x >= half;
  const int w0 = left ? wid - nw : wid;
  const int t = SPLIT ? (threadIdx.x & 31) : left ? threadIdx.x - half : threadIdx.x, sp = fx_spin_of(t);
  const int64_t V = L.g.V, x0 = blockIdx.x * (int64_t)(SPLIT ? 16 : half >> 1) + fx_site_of(t), x = min(x0, V - 1);
  const int src = blockIdx.y;
  FxStage& S = stage[wid];
  zd v[1] = {mk(0.0, 0.0)};
  const bool first = !SPLIT || w0 == 0;
  const bool go = L.sc[src].err == 0, live = go && x0 < V && first;   // go: the whole block
  FxH o, w;
  if (go) {
    const FxField f = fx_src(left ? L.fs : L.fr, src, L.vs);
    const zd sc = left ? L.sc[src].sw : L.sc[src].sv;
    if ((threadIdx.x & (half - 1)) < 2) {
      const double q = (threadIdx.x & 1) ? -L.kappa : 1.0;
      cs[left][threadIdx.x & 1] = fx_coef(mk(q * sc.re, q * sc.im));
    }
    __syncthreads();
    FxHalf acc;
    const FxField bas = left ? fx_bw(L, src, j) : fx_bv(L, src, j);
    if (first) {
      fx_load(f, x, sp, o);
      fx_zero(acc, 0);
      const bool okv = fx_axpy(acc, cs[left][0], o);
      fx_encode(acc, !okv, w);
      if (live) fx_put(bas, x, sp, w);
    }
    const bool need = !left || need_q;
    bool ok = true;
    fx_zero(acc, 0);
    if (need) {
      const FxSite s(L.g, x);
      const int dg = left ? 1 : 0;
      FxExps ex;
      acc.E = fx_range(ex, f, 0, L.fu, L.g, s, dg);
      ok = acc.E < FX_BAD;
      if (!ok) acc.E = FX_E_BIAS;
      fx_hops(acc, f, 0, L.fu, L.g, s, ex, dg, sp, S, SPLIT ? w0 : 0, SPLIT ? w0 + 1 : 4);
    }
    if (SPLIT) fx_join_warps<true>(acc, stage + (left ? nw : 0), w0, nw);
    if (need && first) {
      fx_encode(acc, !ok, o);
      // (v_j again from memory: held in registers over the hops it costs a block per SM)
      __syncwarp();
      fx_load(bas, x, sp, w);
      const bool okp = h_finish(acc, w, cs[left][1], o);
      fx_encode(acc, !okp, o);
      if (live) fx_put(fx_src(left ? L.fq : L.fp, src, L.vs), x, sp, o);
    }
    if (left && first) fx_row_put(S.row, w);
  }
  __syncthreads();
  if (live && !left) {
    fx_row_get(stage[wid + nw].row, w);
    v[0] = fx_dot(w, o);
  }
  zd* part = L.part + src * L.part_stride;
  fx_block_partials(v, sum, part, SPLIT ? 1 : nw);
  // (two warps: the block of the unsplit form on the lattices that may be split)
  alpha_finish(L, src, j, part, scratch, SPLIT ? 2 : blockDim.x >> 5);
}

void fx_tsl_stencil(const Lat<double>& L, int j, int need_q, cudaStream_t st) {
  if (fx_split_exact(L)) {
    fx_launch<k_fx_tsl<1>>(dim3(nblocks(L.g.V, 16), L.nsrc), 256, 8 * sizeof(FxStage), st, L, j, need_q);
    return;
  }
  const int sx = two_sided_sites(L);
  fx_launch<k_fx_tsl<0>>(dim3(nblocks(L.g.V, sx), L.nsrc), 4 * sx, (sx / 8) * sizeof(FxStage), st, L, j, need_q);
}

// r = p - alpha_j v_j - beta_j v_{j-1};  s = q - conj(alpha_j) w_j - delta_j w_{j-1}.  The two
// halves of a block's threads form r and s of the same SX (16 or 32) sites; s crosses to
// the first half for s^dag r.
// Bound by the latency of its loads and of the closing sums: 26 us at 14x14^3 (40 in FP64),
// of which its bytes take 9 and the sums and scalars 8.
// v[0] = s^dag r, v[1] = (|r|^2, |s|^2)
template <int NT>
__device__ __forceinline__ void omega_finish(const Lat<double>& L, int src, int j, int slot, const zd (&v)[2],
                                             FxSumBuf<2, NT>& sum, zd* scratch) {
  zd* part = L.part + src * L.part_stride;
  fx_block_partials(v, sum, part, blockDim.x >> 5);
  if (arrive_last(L.cnt + src * 16 + slot, gridDim.x)) {
    zd s[2];
    fx_sum_partials<2>(part, gridDim.x, s, scratch, blockDim.x >> 5);
    if (threadIdx.x < 32 && L.sc[src].err == 0) omega_finalize_warp(L, src, j, s[0], s[1].re, s[1].im);
  }
}
__global__ void __launch_bounds__(128, 4) k_fx_update(const __grid_constant__ Lat<double> L, int j, int finalize) {
  __shared__ FxSumBuf<2, 128> sum;
  __shared__ zd scratch[2 * 32];
  __shared__ FxRow rows[2];
  __shared__ FxCoef cs[2][2];
  const int half = blockDim.x >> 1;
  const int left = threadIdx.x >= half;
  const int t = left ? threadIdx.x - half : threadIdx.x, sp = fx_spin_of(t);
  const int64_t V = L.g.V;
  const int src = blockIdx.y;
  zd v[2] = {mk(0.0, 0.0), mk(0.0, 0.0)};
  const bool go = L.sc[src].err == 0;   // the whole block
  if (go && t == 0) {
    const int64_t o = (int64_t)src * L.k + j;
    const zd al = L.alpha[o];
    cs[left][0] = fx_coef(left ? -conj(al) : -al);
    cs[left][1] = fx_coef(j == 0 ? mk(0.0, 0.0) : left ? mk(-L.delta[o], 0.0) : -L.beta[o]);
  }
  __syncthreads();
  const int64_t per = half >> 1;
  for (int64_t b = blockIdx.x; go && b * per < V; b += gridDim.x) {
    const int64_t x0 = b * per + fx_site_of(t), x = min(x0, V - 1);
    FxH f;
    FxHalf acc;
    fx_zero(acc, 0);
    fx_load(fx_src(left ? L.fq : L.fp, src, L.vs), x, sp, f);
    bool ok = fx_add(acc, f);
    // what is left of p below 2^-53 of it is its coefficients' rounding: an exact breakdown
    // (r = 0) stays one
    const int zero_top = f.e + 1078 - 53;
    fx_load(left ? fx_bw(L, src, j) : fx_bv(L, src, j), x, sp, f);
    ok = fx_axpy(acc, cs[left][0], f) && ok;
    if (j > 0) {
      fx_load(left ? fx_bw(L, src, j - 1) : fx_bv(L, src, j - 1), x, sp, f);
      ok = fx_axpy(acc, cs[left][1], f) && ok;
    }
    fx_encode(acc, !ok, f, zero_top);
    if (x0 < V) fx_put(fx_src(left ? L.fs : L.fr, src, L.vs), x, sp, f);
    if (!finalize) continue;
    if (left) fx_row_put(rows[t >> 5], f);
    __syncthreads();
    if (x0 < V) {
      if (left) {
        v[1].im += fx_norm2(f);
      } else {
        FxH s;
        fx_row_get(rows[t >> 5], s);
        v[0] = v[0] + fx_dot(s, f);
        v[1].re += fx_norm2(f);
      }
    }
    __syncthreads();
  }
  if (finalize) omega_finish(L, src, j, 2, v, sum, scratch);
}
void fx_tsl_update(const Lat<double>& L, int j, int finalize, cudaStream_t st) {
  const int sx = two_sided_sites(L);
  k_fx_update<<<dim3(one_wave(L, sx), L.nsrc), 4 * sx, 0, st>>>(L, j, finalize);
}

// ---------------------------------------------------------------------------
// Gram-Schmidt projections
// ---------------------------------------------------------------------------
// conj(b) a over all twelve components of a site: |hh| < 24 2^54, |x| < 48 2^56
struct FxS {
  int4 q[12];
  int e;
};
__device__ __forceinline__ void fx_load_site(const FxField& f, int64_t s, FxS& o) {
  const int4* p = f.c + fx_at(s);
#pragma unroll
  for (int i = 0; i < 12; ++i) o.q[i] = p[i * 32];
  o.e = f.e[s];
}
constexpr int FX_NB = 8;   // basis vectors per block
// One thread per site (spt sites in turn), one side per block: side 0 dots W with a, side 1
// V with b.  a's integers stay in registers while FX_NB basis vectors stream past; each
// thread's FP64 sums live in shared memory, so the loop over them stays rolled.  Bound by HBM:
// 56 ms of dots per call at 14x14^3, k = 800 (148 in FP64, at 87% of its units' rate; the
// basis vectors' bytes take 48.5).
__global__ void __launch_bounds__(128, 3) k_fx_dots(const __grid_constant__ Lat<double> L, int nb, FxField a, FxField b,
                                                    int64_t ab_stride, zd* __restrict__ cpart, int64_t cp_stride,
                                                    int spt) {
  __shared__ zd acc[FX_NB][128];
  __shared__ double red[4][2 * FX_NB];
  const int src = blockIdx.z >> 1, side = blockIdx.z & 1;
  const int i0 = blockIdx.y * FX_NB, n = min(FX_NB, nb - i0);
  const int64_t V = L.g.V;
  const FxField f = fx_src(side ? b : a, src, ab_stride);
  for (int i = 0; i < n; ++i) acc[i][threadIdx.x] = mk(0.0, 0.0);
  for (int q = 0; q < spt; ++q) {
    const int64_t x = (blockIdx.x * (int64_t)spt + q) * 128 + threadIdx.x;
    if (x >= V) break;
    FxS u;
    fx_load_site(f, x, u);
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
      FxS w;
      fx_load_site(side ? fx_bv(L, src, i0 + i) : fx_bw(L, src, i0 + i), x, w);
      FxAcc t{0, 0, 0, 0};
#pragma unroll
      for (int c = 0; c < 12; ++c) fx_cdot(t, w.q[c], u.q[c]);
      const double un = w.e == FX_BAD || u.e == FX_BAD ? fx_nan() : fx_pow2_wide(w.e + u.e - 2158 + 57);
      zd s = acc[i][threadIdx.x];
      s.re = fma(un, (double)((t.hr << 3) + (t.xr >> 27)), s.re);
      s.im = fma(un, (double)((t.hi << 3) + (t.xi >> 27)), s.im);
      acc[i][threadIdx.x] = s;
    }
  }
  double v[2 * FX_NB];
#pragma unroll
  for (int i = 0; i < FX_NB; ++i) {
    const zd s = i < n ? acc[i][threadIdx.x] : mk(0.0, 0.0);
    v[2 * i] = s.re;
    v[2 * i + 1] = s.im;
  }
  const double s = warp_sum_multi(v);
  const int lane = threadIdx.x & 31;
  if (!(lane & 1)) red[threadIdx.x >> 5][lane >> 1] = s;
  __syncthreads();
  if (threadIdx.x < 2 * n) {
    double r = red[0][threadIdx.x];
    for (int w = 1; w < 4; ++w) r = r + red[w][threadIdx.x];
    reinterpret_cast<double*>(cpart + src * cp_stride + (int64_t)(2 * (i0 + threadIdx.x / 2) + side) * gridDim.x +
                              blockIdx.x)[threadIdx.x & 1] = r;
  }
}
// one warp per coefficient: its site blocks' partials in lane-strided order, then a fixed tree
__global__ void __launch_bounds__(128) k_fx_dots_reduce(const zd* __restrict__ cpart, int64_t cp_stride, int nsb, int nb,
                                                        zd* __restrict__ coef, int64_t coef_stride) {
  const int i = (blockIdx.x * 4 + (threadIdx.x >> 5)), lane = threadIdx.x & 31;
  const int src = blockIdx.y;
  if (i >= 2 * nb) return;
  const zd* cp = cpart + src * cp_stride + (int64_t)i * nsb;
  zd s = mk(0.0, 0.0);
  for (int b = lane; b < nsb; b += 32) s = s + cp[b];
  s = warp_sum(s);
  if (lane == 0) coef[src * coef_stride + i] = s;
}
void fx_proj_dots(const Lat<double>& L, int nb, const FxField& a, const FxField& b, int64_t ab_stride, zd* coef,
                  zd* cpart, cudaStream_t st) {
  // four sites per thread from V = 32768 on (the block's reduction then costs a quarter per site)
  const int spt = L.g.V >= 32768 ? 4 : 1;
  const unsigned nsb = nblocks(L.g.V, 128 * spt);
  const int64_t cp_stride = (int64_t)2 * L.k * nsb;
  k_fx_dots<<<dim3(nsb, nblocks(nb, FX_NB), 2 * L.nsrc), 128, 0, st>>>(L, nb, a, b, ab_stride, cpart, cp_stride, spt);
  k_fx_dots_reduce<<<dim3(nblocks(2 * nb, 4), L.nsrc), 128, 0, st>>>(cpart, cp_stride, nsb, nb, coef, 2 * (int64_t)L.k);
}

// A long sum of coefficient times field, kept as (hh, x) pairs: per term only the products,
// the coefficient being shifted to the sum's scale.  A term adds less than 2^57 to hh and
// 2^59.4 to x: x is folded into hh after eight, and hh scaled down when it may pass 2^60.
struct FxTerms {
  FxAcc t[6];
  int E, n;
  bool ok;
  __device__ __forceinline__ void init() {
#pragma unroll
    for (int i = 0; i < 6; ++i) t[i] = FxAcc{0, 0, 0, 0};
    E = 0;
    n = 0;
    ok = true;
  }
  __device__ __forceinline__ void fold() {
    int m = 0;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      t[i].hr += (t[i].xr + (1ll << 29)) >> 30;
      t[i].hi += (t[i].xi + (1ll << 29)) >> 30;
      t[i].xr = t[i].xi = 0;
      m |= fx_top(FxZ{t[i].hr, t[i].hi});
    }
    n = 0;
    if (m >= (1 << 28)) down(2);
  }
  __device__ __forceinline__ void down(int sh) {
    const fxll r = (1ll << sh) >> 1;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      t[i].hr = (t[i].hr + r) >> sh;
      t[i].hi = (t[i].hi + r) >> sh;
      t[i].xr = (t[i].xr + r) >> sh;
      t[i].xi = (t[i].xi + r) >> sh;
    }
    E += sh;
  }
  __device__ __forceinline__ void add(const FxCoef& c, const FxH& f) {
    if (f.e == FX_BAD || c.e == FX_BAD) {
      ok = false;
      return;
    }
    const int et = f.e + c.e;
    if (et > E) {
      down(min(et - E, 62));
      E = et;
    }
    const int d = E - et;
    if (d > 59) return;
    const fxll half = (1ll << d) >> 1;
    const FxInt a = fx_split((fx_join(c.c.x, c.c.y) + half) >> d), b = fx_split((fx_join(c.c.z, c.c.w) + half) >> d);
    const int4 k = make_int4(a.h, a.l, b.h, b.l);
#pragma unroll
    for (int i = 0; i < 6; ++i) fx_cmac(t[i], k, f.q[i]);
    if (++n == 8) fold();
  }
  // the sum, below 2^60.6 units
  __device__ __forceinline__ void value(FxHalf& o) {
    fold();
#pragma unroll
    for (int i = 0; i < 6; ++i) o.v[i] = FxZ{t[i].hr, t[i].hi};
    o.E = E;
  }
};
// a -= b (a below 2^61, b below 2^60.6 units of their scales)
__device__ __forceinline__ void fx_subtract(FxHalf& a, FxHalf& b) {
  if (b.E > a.E) fx_raise(a, b.E);
  const int sh = min(a.E - b.E, 62);
  const fxll r = (1ll << sh) >> 1;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    a.v[i].re -= (b.v[i].re + r) >> sh;
    a.v[i].im -= (b.v[i].im + r) >> sh;
  }
}

constexpr int FX_CH = 12;   // coefficients converted at a time per side (a multiple of 4 FX_RING)
// T += sum_i coef[ci + cstep i] u_i(x) over nb vectors; the coefficients are converted by the
// nt threads of a group (t = 0 .. nt - 1), one chunk ahead of their use, in cs[0] and cs[1].
// Every thread of the block calls this with the same nb.
template <typename At>
__device__ __forceinline__ void sum_vectors(FxTerms& T, FxStage& S, FxCoef (*cs)[FX_CH], const zd* coef, int cstep,
                                            int nb, int64_t x, int sp, int t, int nt, const At& at0, int w = 0,
                                            int nw = 1) {
  FxStream q;
  // this warp's vectors: i = w, w + nw, ...
  const int nv = (nb - w + nw - 1) / nw;
  const auto at = [&](int i) { return at0(w + i * nw); };
  for (int i = t; i < min(FX_CH, nb); i += nt) cs[0][i] = fx_coef(coef[(int64_t)i * cstep]);
  q.start(S, nv, x, sp, at);
  int v0 = 0;   // this warp's first vector of the chunk
  for (int i0 = 0, c = 0; i0 < nb; i0 += FX_CH, c ^= 1) {
    __syncthreads();   // this chunk's coefficients are there, and the last chunk's are done with
    for (int i = i0 + FX_CH + t; i < min(i0 + 2 * FX_CH, nb); i += nt)
      cs[c ^ 1][i - i0 - FX_CH] = fx_coef(coef[(int64_t)i * cstep]);
    const int v1 = min((i0 + FX_CH - w + nw - 1) / nw, nv);
#pragma unroll 1
    for (int v = v0; v < v1; v += FX_RING) {
#pragma unroll
      for (int u = 0; u < FX_RING; ++u) {
        if (v + u < v1) {
          FxH f;
          q.next(S, u, v + u, nv, x, sp, at, f);
          T.add(cs[c][w + (v + u) * nw - i0], f);
        }
      }
    }
    v0 = v1;
  }
  fx_copy_wait<0>();
}

// a -= sum_i coefA_i v_i by the first half of a block's threads, b -= sum_i coefB_i w_i by
// the second, for the same SX sites.  fin: omega and the next scales (a = r, b = s).
//
// SPLIT: on a lattice with too few sites to fill the GPU four warps share a side's 16 sites,
// a quarter of the vectors each (88 us per projection of 100 vectors at 4^4 without, 36 with).
// Above 16 sites per SM the joins cost more than they give (6x12^3: 95 ms per call, 114 split).
// Bound by HBM: 58 ms per call at 14x14^3, k = 800 (146 in FP64; the bytes take 48.5).
template <int SPLIT>
__global__ void __launch_bounds__(SPLIT ? 256 : 128, SPLIT ? 1 : 3)
    k_fx_proj_update(const __grid_constant__ Lat<double> L, int nb, FxField a, FxField b, int64_t ab_stride,
                     const zd* __restrict__ coef, int64_t coef_stride, int j, int fin) {
  constexpr int NT = SPLIT ? 256 : 128;
  extern __shared__ __align__(16) unsigned char fx_smem[];
  FxStage* stage = reinterpret_cast<FxStage*>(fx_smem);
  FxSumBuf<2, NT>& sum2 = *reinterpret_cast<FxSumBuf<2, NT>*>(fx_smem);
  __shared__ FxCoef cs[2][2][FX_CH];
  __shared__ zd scratch[2 * 32];
  const int half = blockDim.x >> 1, wid = threadIdx.x >> 5, nw = half >> 5;   // nw warps per side
  const int left = threadIdx.x >= half;
  const int w0 = left ? wid - nw : wid, th = left ? threadIdx.x - half : threadIdx.x;
  const int t = SPLIT ? (threadIdx.x & 31) : th, sp = fx_spin_of(t);
  const int64_t V = L.g.V, x0 = blockIdx.x * (int64_t)(SPLIT ? 16 : half >> 1) + fx_site_of(t), x = min(x0, V - 1);
  const int src = blockIdx.y;
  FxStage& S = stage[wid];
  const bool first = !SPLIT || w0 == 0;
  const bool live = x0 < V && first;
  FxTerms T;
  T.init();
  const FxField u0 = left ? fx_bw(L, src, L.jbase) : fx_bv(L, src, L.jbase);
  sum_vectors(T, S, cs[left], coef + src * coef_stride + left, 2, nb, x, sp, th, half,
              [&](int i) { return fx_src(u0, i - L.jbase, L.vs); }, SPLIT ? w0 : 0, SPLIT ? 4 : 1);
  const FxField fa = fx_src(left ? b : a, src, ab_stride);
  FxH f;
  {
    FxHalf acc, s;
    T.value(s);
    bool ok = T.ok;
    if (SPLIT) {
      if (!ok) s.E = FX_BAD;   // a marked site of any warp's vectors marks the sum
      fx_join_warps<false>(s, stage + (left ? nw : 0), w0, nw);
      ok = s.E < FX_BAD;
    }
    if (first) {
      fx_load(fa, x, sp, f);
      fx_zero(acc, 0);
      ok = fx_add(acc, f) && ok;
      fx_subtract(acc, s);
      fx_encode(acc, !ok, f);
      if (live) fx_put(fa, x, sp, f);
    }
  }
  if (!fin) return;
  __syncthreads();   // the stages are done with
  zd v[2] = {mk(0.0, 0.0), mk(0.0, 0.0)};
  if (left && first) fx_row_put(S.row, f);
  __syncthreads();
  if (live) {
    if (left) {
      v[1] = mk(0.0, fx_norm2(f));
    } else {
      FxH s;
      fx_row_get(stage[wid + nw].row, s);
      v[0] = fx_dot(s, f);
      v[1] = mk(fx_norm2(f), 0.0);
    }
  }
  __syncthreads();
  omega_finish(L, src, j, 3, v, sum2, scratch);
}
void fx_proj_update(const Lat<double>& L, int nb, const FxField& a, const FxField& b, int64_t ab_stride, const zd* coef,
                    int j, int fin, cudaStream_t st) {
  const int64_t cs = 2 * (int64_t)L.k;
  if (L.g.V < 152 * 16) {   // fewer than two warps per SM without the split
    fx_launch<k_fx_proj_update<1>>(dim3(nblocks(L.g.V, 16), L.nsrc), 256, 8 * sizeof(FxStage), st, L, nb, a, b, ab_stride,
                                   coef, cs, j, fin);
    return;
  }
  fx_launch<k_fx_proj_update<0>>(dim3(nblocks(L.g.V, 32), L.nsrc), 128, 4 * sizeof(FxStage), st, L, nb, a, b, ab_stride,
                                 coef, cs, j, fin);
}

// out[src] (+)= sum_{j0 <= i < j0 + nvec} y_i u_i in the user's layout, u = V (side 0) or W;
// y at ystride per source, sources src0, src0 + 1, ...
__global__ void __launch_bounds__(128, 3) k_fx_combine(const __grid_constant__ Lat<double> L, int src0, int side, int j0,
                                                       int nvec, const zd* __restrict__ y, int64_t ystride,
                                                       double* __restrict__ out, int accumulate) {
  __shared__ FxStage stage[4];
  __shared__ FxCoef cs[2][FX_CH];
  const int sp = fx_spin_of(threadIdx.x), w = threadIdx.x >> 5;
  const int64_t V = L.g.V, xw = blockIdx.x * (int64_t)(blockDim.x >> 1) + w * 16;
  const int64_t x = min(xw + (threadIdx.x & 15), V - 1);
  FxTerms T;
  T.init();
  const int src = src0 + blockIdx.y;
  const FxField u0 = side ? fx_bw(L, src, j0) : fx_bv(L, src, j0);
  sum_vectors(T, stage[w], cs, y + blockIdx.y * ystride + j0, 1, nvec, x, sp, threadIdx.x, blockDim.x,
              [&](int i) { return fx_src(u0, i, L.vs); });
  if (xw >= V) return;   // whole warps
  FxHalf s;
  T.value(s);
  zd o[6];
  fx_double(s, !T.ok, o);
  __syncwarp();
  if (accumulate) {
    zd p[6];
    aos_load(out, blockIdx.y, V, xw, stage[w].out, sp, p);
#pragma unroll
    for (int i = 0; i < 6; ++i) o[i] = p[i] + o[i];
  }
  aos_store(out, blockIdx.y, V, xw, stage[w].out, sp, o);
}
void fx_combine(const Lat<double>& L, int src0, int nsrc, int side, int j0, int nvec, const zd* y, int64_t ystride,
                double* out, int accumulate, cudaStream_t st) {
  const int bs = L.g.V < 152 * 64 ? 32 : 128;
  k_fx_combine<<<dim3(nblocks(L.g.V, bs / 2), nsrc), bs, 0, st>>>(L, src0, side, j0, nvec, y, ystride, out,
                                                                  accumulate);
}

}  // namespace ov
