// FP64 stencil kernels in block fixed point (fx.cuh): ov_apply_H, the two-sided
// Lanczos step's H / H^dagger pair (plain and Theorem-1 block form) and the
// reverse sweep's stencil.  Each falls back, site by site, to FP64 arithmetic
// where the fixed-point form does not hold.
#include "fx.cuh"
#include "kernels.h"
#include "recurrence.cuh"

namespace ov {

static inline unsigned nblocks(int64_t n, int bs) { return (unsigned)((n + bs - 1) / bs); }

// ---------------------------------------------------------------------------
// links in fixed point
// ---------------------------------------------------------------------------
// Direction d = blockIdx.y: the links (d < 3 spatial, 3: ef U_t, 4: efinv U_t) of the
// user's array u, or with dh the combinations of the directional derivative dH:
// d < 3: E, 3: ef (E_t + m U_t), 4: efinv (E_t - m U_t), E (may be null: zero) in e.
// The products are formed with their FP64 rounding errors, so each entry carries the
// fixed-point error alone.
__global__ void __launch_bounds__(128) k_pack_links_fx(const double* __restrict__ u, const double* __restrict__ e,
                                                       int dh, double m, double ef, double efinv,
                                                       int4* __restrict__ out, short* __restrict__ ex, int64_t V) {
  const int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (x >= V) return;
  const int d = blockIdx.y, nu = d < 3 ? d : 3;
  const double f = d < 3 ? 1.0 : (d == 3 ? ef : efinv);
  const double2* iu = reinterpret_cast<const double2*>(u) + x * 36 + nu * 9;
  const double2* ie = e ? reinterpret_cast<const double2*>(e) + x * 36 + nu * 9 : nullptr;
  const double mm = d == 3 ? m : -m;
  double hi[18], lo[18];
  unsigned mag = 0u;
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    double2 a, al = make_double2(0.0, 0.0);
    if (!dh) {
      a = iu[q];
    } else {
      a = ie ? ie[q] : make_double2(0.0, 0.0);
      if (d >= 3) {   // E + mm U, as a sum and its rounding error
        const double2 t = iu[q];
        const double pr = mm * t.x, pi = mm * t.y;
        const double er = fma(mm, t.x, -pr), ei = fma(mm, t.y, -pi);
        const double sr = a.x + pr, si = a.y + pi;
        const double zr = sr - a.x, zi = si - a.y;
        al.x = ((a.x - (sr - zr)) + (pr - zr)) + er;
        al.y = ((a.y - (si - zi)) + (pi - zi)) + ei;
        a = make_double2(sr, si);
      }
    }
    if (d < 3) {
      hi[2 * q] = a.x;
      hi[2 * q + 1] = a.y;
      lo[2 * q] = lo[2 * q + 1] = 0.0;
    } else {
      hi[2 * q] = f * a.x;
      hi[2 * q + 1] = f * a.y;
      lo[2 * q] = fma(f, a.x, -hi[2 * q]) + f * al.x;
      lo[2 * q + 1] = fma(f, a.y, -hi[2 * q + 1]) + f * al.y;
    }
    mag = max(mag, max(fx_mag(hi[2 * q]), fx_mag(hi[2 * q + 1])));
  }
  const int eb = (int)(mag >> 20);
  const bool bad = mag != 0u && (eb < FX_U_MIN || eb > FX_U_MAX);
  const int ee = mag == 0u ? 1022 : eb;
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
    out[(int64_t)(d * 9 + q) * V + x] = make_int4(r.h, r.l, i.h, i.l);
  }
}
void pack_links_fx(const double* u, int4* out, short* ex, int64_t V, double ef, double efinv, cudaStream_t st) {
  k_pack_links_fx<<<dim3(nblocks(V, 128), 5), 128, 0, st>>>(u, nullptr, 0, 0.0, ef, efinv, out, ex, V);
}
void pack_dh_links_fx(const double* u, const double* e, double m, int4* out, short* ex, int64_t V, double ef,
                      double efinv, cudaStream_t st) {
  k_pack_links_fx<<<dim3(nblocks(V, 128), 5), 128, 0, st>>>(u, e, 1, m, ef, efinv, out, ex, V);
}

// ---------------------------------------------------------------------------
// encoding FP64 fields
// ---------------------------------------------------------------------------
// user spinors [src][site][12] to fixed point; FP64 values (site-major) only where a site
// is out of the window
__global__ void __launch_bounds__(128) k_fx_pack(const double* __restrict__ aos, FxField f, double* __restrict__ d,
                                                 int64_t V, int64_t vs) {
  const int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int src = blockIdx.y;
  if (x >= V) return;
  const double2* in = reinterpret_cast<const double2*>(aos) + ((int64_t)src * V + x) * 12;
  Spinor<double> p;
#pragma unroll
  for (int c = 0; c < 12; ++c) {
    const double2 t = in[c];
    p.c[c] = mk(t.x, t.y);
  }
  if (fx_store(fx_src(f, src, vs, V), V, x, p)) store_spinor(d + src * vs, V, x, p);
}
void fx_pack(const double* aos, const FxField& f, double* d, int nsrc, int64_t V, int64_t vs, cudaStream_t st) {
  k_fx_pack<<<dim3(nblocks(V, 128), nsrc), 128, 0, st>>>(aos, f, d, V, vs);
}
__global__ void __launch_bounds__(128) k_fx_encode(const double* __restrict__ d, FxField f, int64_t V, int64_t vs) {
  const int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int src = blockIdx.y;
  if (x >= V) return;
  Spinor<double> p;
  load_spinor_ro(d + src * vs, V, x, p);
  fx_store(fx_src(f, src, vs, V), V, x, p);
}
void fx_encode(const double* d, const FxField& f, int nsrc, int64_t V, int64_t vs, cudaStream_t st) {
  k_fx_encode<<<dim3(nblocks(V, 128), nsrc), 128, 0, st>>>(d, f, V, vs);
}

// ---------------------------------------------------------------------------
// the site's hop sum a with out = psi - kappa a (upper spins), kappa a - psi (lower)
// ---------------------------------------------------------------------------
// FP64 form (out of line: reached only where a site or link is out of its window)
__device__ __noinline__ void hops_fp64(const FxLoad& ld, const double* u, const Geom& g, int64_t x, double ft,
                                       double fti, Spinor<double>* a) {
  int c[4];
  site_coords(g, x, c);
  Spinor<double> t;
  spinor_zero(t);
  hop_dir<0>(t, ld, u, g, x, c, ft, fti);
  hop_dir<1>(t, ld, u, g, x, c, ft, fti);
  hop_dir<2>(t, ld, u, g, x, c, ft, fti);
  hop_dir<3>(t, ld, u, g, x, c, ft, fti);
  *a = t;
}
// dH's hop sum added to a (dh_site_ld's result is -kappa times it on the upper spins)
__device__ __noinline__ void dh_hops_fp64_add(const FxLoad& ld, const double* ue, const double* u, const Geom& g,
                                              int64_t x, double ft, double fti, double m, Spinor<double>* a) {
  Spinor<double> t;
  dh_site_ld(ld, ue, u, g, x, 1.0, ft, fti, m, t);
  for (int i = 0; i < 12; ++i) a->c[i] = i < 6 ? a->c[i] - t.c[i] : a->c[i] + t.c[i];
}
__device__ __forceinline__ void fx_double(const FxHalf& s, zd (&a)[6]) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    a[i] = mk((double)s.up[i].re, (double)s.up[i].im);
    a[3 + i] = mk((double)s.lo[i].re, (double)s.lo[i].im);
  }
}
// the thread's six components of the hop sum of fixed-point field f, in units of the returned
// power of two (1 from the FP64 form); d: the field's FP64 companion.  Every lane of the warp.
__device__ __forceinline__ double hop_sum(const Lat<double>& L, const FxField& f, const double* d, int64_t x,
                                          int dagger, int sp, bool live, zd (&a)[6]) {
  FxHalf acc;
  fx_zero(acc);
  int E = 0;
  if (live) {
    const FxSite s(L.g, x);
    fx_range(E, f, 0, L.fu, L.g, s, dagger);
    if (E < FX_BAD) fx_hops(acc, E, f, L.g.V, 0, L.fu, L.g, s, dagger, sp);
  }
  fx_exchange(acc);
  if (E >= FX_BAD) {
    Spinor<double> t;
    hops_fp64(FxLoad{f, d, L.g.V, 0}, L.u, L.g, x, dagger ? L.efinv : L.ef, dagger ? L.ef : L.efinv, &t);
    fx_pick(t, sp, a);
    return 1.0;
  }
  fx_double(acc, a);
  return fx_pow2(E - FX_E_BIAS);
}

// thread t of a group of 2 n threads: site t / 32 * 16 + t % 16, spin (t / 16) % 2
__device__ __forceinline__ int fx_site_of(int t) { return (t >> 5) * 16 + (t & 15); }
__device__ __forceinline__ int fx_spin_of(int t) { return (t >> 4) & 1; }

// ---------------------------------------------------------------------------
// ov_apply_H: two threads per (site, source); blocks of blockDim.x / 2 sites x blockDim.y
// sources, whose sources share the link loads through L1.  With aos the output is the
// user's layout, written through shared memory (a warp's 16 sites are 3 KB in a row).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(128, 4) k_fx_apply(const __grid_constant__ Lat<double> L, FxField in,
                                                     const double* __restrict__ din, double* __restrict__ out,
                                                     int dagger, int aos) {
  __shared__ double2 stage[4][16 * 13];
  const int sp = fx_spin_of(threadIdx.x);
  const int64_t x0 = blockIdx.x * (int64_t)(blockDim.x >> 1) + (threadIdx.x >> 5) * 16, x = x0 + (threadIdx.x & 15);
  const int src = blockIdx.y * blockDim.y + threadIdx.y;
  const int64_t V = L.g.V;
  if (src >= L.nsrc || x0 >= V) return;   // whole warps
  const bool live = x < V;
  const FxField f = fx_src(in, src, L.vs, V);
  const double* d = din + (int64_t)src * L.vs;
  zd a[6];
  const double ks = L.kappa * hop_sum(L, f, d, x, dagger, sp, live, a);
  if (live) {
    const int e = f.e[x];
    const double u = e == FX_BAD ? 1.0 : fx_pow2(e - 1079);
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      const int c = (i < 3 ? sp * 3 + i : (2 + sp) * 3 + i - 3);
      zd p;
      if (e == FX_BAD) {
        const double2 t = reinterpret_cast<const double2*>(d)[c * V + x];
        p = mk(t.x, t.y);
      } else {
        p = u * fx_value(__ldg(f.c + c * V + x));
      }
      const zd q = mk(fma(-ks, a[i].re, p.re), fma(-ks, a[i].im, p.im));
      a[i] = i < 3 ? q : -q;
    }
  }
  if (!aos) {
    if (live) fx_store_half(out + (int64_t)src * L.vs, V, x, sp, a);
    return;
  }
  double2* st = stage[(threadIdx.y * blockDim.x + threadIdx.x) >> 5];
  const int lane = threadIdx.x & 31, ns = (int)min((int64_t)16, V - x0);
#pragma unroll
  for (int i = 0; i < 6; ++i)
    st[(lane & 15) * 13 + (i < 3 ? sp * 3 + i : (2 + sp) * 3 + i - 3)] = make_double2(a[i].re, a[i].im);
  __syncwarp();
  double2* o = reinterpret_cast<double2*>(out) + ((int64_t)src * V + x0) * 12;
  for (int i = lane; i < ns * 12; i += 32) o[i] = st[i / 12 * 13 + i % 12];
}
void fx_apply_h(const Lat<double>& L, const FxField& in, const double* d, double* out, int dagger, int aos,
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
  k_fx_apply<<<dim3(nblocks(L.g.V, sx / 2), nblocks(L.nsrc, sy)), dim3(sx, sy), 0, st>>>(L, in, d, out, dagger, aos);
}

// ---------------------------------------------------------------------------
// TSL step j (see k_tsl_stencil): v_j = sv r, w_j = sw s, p = H v_j, q = H^dag w_j,
// alpha_j = w_j^dag p.  A block of 4 SX threads covers SX (16 or 32) sites; its first
// half of warps forms v_j and p, the second half w_j and q of the same sites, so the
// links of both products come from L1 and a small lattice spreads over more warps.
// w_j crosses to the first half through shared memory for the dot product.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void alpha_finish(const Lat<double>& L, int src, int j, zd (&v)[1], zd* scratch) {
  block_sum<1>(v, scratch);
  zd* part = L.part + src * L.part_stride;
  if (threadIdx.x == 0) part[blockIdx.x] = v[0];
  if (arrive_last(L.cnt + src * 16 + 1, gridDim.x)) {
    zd s[1];
    sum_partials<1>(part, gridDim.x, s, scratch);
    if (threadIdx.x == 0) {
      SrcScal& sc = L.sc[src];
      if (!finite_z(s[0])) flag_error(sc, ERRB_NONFINITE, j);
      L.alpha[(int64_t)src * L.k + j] = s[0];
    }
  }
}
// +-(p - kc a): the thread's six components of sc (H psi) from p = sc psi, a the hop sum, kc = kappa sc
__device__ __forceinline__ void h_finish(zd (&p)[6], const zd (&a)[6], zd kc) {
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    zd q = mk(fma(-kc.re, a[i].re, p[i].re), fma(-kc.re, a[i].im, p[i].im));
    if (kc.im != 0.0) q = mk(fma(kc.im, a[i].im, q.re), fma(-kc.im, a[i].re, q.im));
    p[i] = i < 3 ? q : -q;
  }
}

__global__ void __launch_bounds__(128, 4) k_fx_tsl(const __grid_constant__ Lat<double> L, int j, int need_q) {
  __shared__ zd scratch[32];
  __shared__ double2 ws[6][64];
  const int half = blockDim.x >> 1;
  const bool left = threadIdx.x >= half;
  const int t = left ? threadIdx.x - half : threadIdx.x, sp = fx_spin_of(t);
  const int64_t x = blockIdx.x * (int64_t)(half >> 1) + fx_site_of(t);
  const int src = blockIdx.y;
  const int64_t V = L.g.V;
  zd v[1] = {mk(0.0, 0.0)};
  const bool live = x < V && L.sc[src].err == 0;
  zd o[6], a[6];
  const double* d = (left ? L.s : L.r) + src * L.vs;
  double* bas = left ? L.basis_w(src, j) : L.basis_v(src, j);
  const zd sc = left ? L.sc[src].sw : L.sc[src].sv;
  double unit = 0.0;
  if (!left || need_q)
    unit = hop_sum(L, fx_src(left ? L.fs : L.fr, src, L.vs, V), d, x, left ? 1 : 0, sp, live, a);
  if (live) {
    fx_load_half(d, V, x, sp, o);
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      o[c] = sc.im != 0.0 ? sc * o[c] : mk(sc.re * o[c].re, sc.re * o[c].im);
      if (left) ws[c][t] = make_double2(o[c].re, o[c].im);
    }
    fx_store_half(bas, V, x, sp, o);
    if (!left || need_q) {
      const double ks = L.kappa * unit;
      h_finish(o, a, mk(ks * sc.re, ks * sc.im));
      fx_store_half((left ? L.q : L.p) + src * L.vs, V, x, sp, o);
    }
  }
  __syncthreads();
  if (live && !left) {
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const double2 w = ws[c][t];
      cdotac(v[0], mk(w.x, w.y), o[c]);
    }
  }
  alpha_finish(L, src, j, v, scratch);
}

// Block step (see k_tsl_stencil_block): four warps of 16 sites,
//   0: p_u = H v_u + dH v_l   1: p_l = H v_l   2: q_u = H^dag w_u   3: q_l = dH^dag w_u + H^dag w_l
__global__ void __launch_bounds__(128, 4) k_fx_tsl_block(const __grid_constant__ Lat<double> L, int j, int need_q) {
  __shared__ zd scratch[32];
  __shared__ double2 ws[2][6][32];
  const int t = threadIdx.x & 31, part_id = threadIdx.x >> 5, sp = fx_spin_of(t);
  const bool left = part_id >= 2, low = part_id & 1;
  const int64_t x = blockIdx.x * (int64_t)16 + fx_site_of(t);
  const int src = blockIdx.y;
  const int64_t V = L.gl.V, Vf = L.g.V;
  const int off = low ? (int)V : 0, offx = low ? 0 : (int)V;
  const bool cross = part_id == 0 || part_id == 3;   // adds dH of the other half
  zd v[1] = {mk(0.0, 0.0)};
  const bool live = x < V && L.sc[src].err == 0;
  zd o[6], a[6];
  const double* d = (left ? L.s : L.r) + src * L.vs;
  double* bas = left ? L.basis_w(src, j) : L.basis_v(src, j);
  const zd sc = left ? L.sc[src].sw : L.sc[src].sv;
  double unit = 0.0;
  if (!left || need_q) {
    const FxField f = fx_src(left ? L.fs : L.fr, src, L.vs, Vf);
    const int dg = left ? 1 : 0;
    FxHalf acc;
    fx_zero(acc);
    int E = 0;
    if (live) {
      const FxSite s(L.gl, x);
      fx_range(E, f, off, L.fu, L.gl, s, dg);
      if (cross) {
        fx_range(E, f, offx, L.fd, L.gl, s, dg);
        ++E;   // sixteen hops
      }
      if (E < FX_BAD)
        for (int h = 0; h < (cross ? 2 : 1); ++h)
          fx_hops(acc, E, f, Vf, h ? offx : off, h ? L.fd : L.fu, L.gl, s, dg, sp);
    }
    fx_exchange(acc);
    if (E < FX_BAD) {
      fx_double(acc, a);
      unit = fx_pow2(E - FX_E_BIAS);
    } else {
      const double ft = left ? L.efinv : L.ef, fti = left ? L.ef : L.efinv;
      Spinor<double> b;
      hops_fp64(FxLoad{f, d, Vf, off}, L.u, L.gl, x, ft, fti, &b);
      if (cross) dh_hops_fp64_add(FxLoad{f, d, Vf, offx}, L.ue, L.u, L.gl, x, ft, fti, left ? -L.mdir : L.mdir, &b);
      fx_pick(b, sp, a);
      unit = 1.0;
    }
  }
  if (live) {
    fx_load_half(d, Vf, off + x, sp, o);
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      o[c] = sc * o[c];
      if (left) ws[low][c][t] = make_double2(o[c].re, o[c].im);
    }
    fx_store_half(bas, Vf, off + x, sp, o);
    if (!left || need_q) {
      const double ks = L.kappa * unit;
      h_finish(o, a, mk(ks * sc.re, ks * sc.im));
      fx_store_half((left ? L.q : L.p) + src * L.vs, Vf, off + x, sp, o);
    }
  }
  __syncthreads();
  if (live && !left) {
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const double2 w = ws[low][c][t];
      cdotac(v[0], mk(w.x, w.y), o[c]);
    }
  }
  alpha_finish(L, src, j, v, scratch);
}

void fx_tsl_stencil(const Lat<double>& L, int j, int need_q, cudaStream_t st, int variant) {
  if (L.block) {
    k_fx_tsl_block<<<dim3(nblocks(L.gl.V, 16), L.nsrc), 128, 0, st>>>(L, j, need_q);
    return;
  }
  const int64_t V = L.g.V;
  // 16 sites per block where 32 would leave SMs without a block
  const int sx = (variant & 1) || V * L.nsrc < 152 * 32 ? 16 : 32;
  k_fx_tsl<<<dim3(nblocks(V, sx), L.nsrc), 4 * sx, 0, st>>>(L, j, need_q);
}

// ---------------------------------------------------------------------------
// Reverse sweep, gradients of v_j and w_j (see k_rev_stencil):
//   Gv_j = H^dag g_p  + sum_i c_i f_i,    Gw_j = H h_in + sum_i c'_i f'_i
// with f over xbar, g_r, the previous g_r and w_{jm+1} of the recorded projections
// (g_s, previous g_s and v_{jm+1} for Gw).  The sums run in the same fixed-point
// accumulator as the hops: with c_i / kappa as coefficients,
//   G = +-(p - kappa [hops -+ sum_i (c_i / kappa) f_i])   (upper / lower spins).
// One half of a block's warps forms Gv, the other Gw, of the same SX (16 or 32) sites.
// The coefficients are converted once per block, RT terms at a time.
// ---------------------------------------------------------------------------
struct RevTerm {
  const double* f;
  zd c;           // coefficient in FP64
  FxCoef k;       // c / kappa
};
// term i of side (0: Gv, 1: Gw) of step j
__device__ __forceinline__ void rev_term(const Lat<double>& L, const Rev<double>& B, int src, int side, int j,
                                         int slot, int prev, int i, RevTerm& t) {
  const int64_t o = (int64_t)src * L.k + j;
  const bool carry = j < L.k - 1, pcarry = prev >= 0 && j + 1 < L.k - 1;
  if (side == 0) {
    if (i == 0) {
      t.f = B.xbar + src * L.vs;
      t.c = conj(B.y[o]);
      return;
    }
    --i;
  }
  if (carry) {
    if (i == 0) {
      t.f = B.ring(side ? B.gs_ring : B.gr_ring, slot, src);
      t.c = side ? -L.alpha[o] : -conj(L.alpha[o]);
      return;
    }
    --i;
  }
  if (pcarry) {
    if (i == 0) {
      t.f = B.ring(side ? B.gs_ring : B.gr_ring, prev, src);
      t.c = side ? mk(-L.delta[o + 1], 0.0) : -conj(L.beta[o + 1]);
      return;
    }
    --i;
  }
  const int jm = B.reb_steps[i];
  const int64_t eo = src * (int64_t)B.nreb_max * L.k + (int64_t)i * L.k + j;
  t.f = side ? L.basis_v(src, jm + 1) : L.basis_w(src, jm + 1);
  t.c = side ? B.ew[eo] : B.ev[eo];
}
// G of one site and side in FP64 (reached only outside the exponent windows)
__device__ __noinline__ void rev_site_fp64(const Lat<double>& L, const Rev<double>& B, int src, int side, int j,
                                           int slot, int prev, int nterms, int64_t x, Spinor<double>* out) {
  const int64_t V = L.g.V;
  const FxLoad ld{fx_src(side ? B.fh : B.fp, src, L.vs, V),
                  side ? B.hin + src * L.vs : B.ring(B.gp_ring, slot, src), V, 0};
  Spinor<double> h, t;
  h_site_ld(ld, L.u, L.g, x, L.kappa, side ? L.ef : L.efinv, side ? L.efinv : L.ef, h);
  for (int i = 0; i < nterms; ++i) {
    RevTerm r;
    rev_term(L, B, src, side, j, slot, prev, i, r);
    load_spinor(r.f, V, x, t);
    for (int c = 0; c < 12; ++c) cmac(h.c[c], r.c, t.c[c]);
  }
  *out = h;
}

constexpr int RT = 16;   // terms converted at a time per side
__global__ void __launch_bounds__(128, 4) k_fx_rev(const __grid_constant__ Lat<double> L,
                                                   const __grid_constant__ Rev<double> B, int j, int slot, int prev,
                                                   int nrec) {
  __shared__ RevTerm terms[2][RT];
  const int half = blockDim.x >> 1;
  const int side = threadIdx.x >= half ? 1 : 0;
  const int t = side ? threadIdx.x - half : threadIdx.x, sp = fx_spin_of(t);
  const int64_t x = blockIdx.x * (int64_t)(half >> 1) + fx_site_of(t);
  const int src = blockIdx.y;
  const int64_t V = L.g.V;
  const int base = (j < L.k - 1 ? 1 : 0) + (prev >= 0 && j + 1 < L.k - 1 ? 1 : 0) + nrec;
  const int nt = base + (side ? 0 : 1), ntmax = base + 1;
  const FxField f = fx_src(side ? B.fh : B.fp, src, L.vs, V);
  const double kinv = 1.0 / L.kappa;
  FxHalf acc;
  fx_zero(acc);
  int E = FX_BAD, ex = FX_BAD;
  bool ok = x < V;
  if (ok) {
    const FxSite s(L.g, x);
    ex = f.e[x];
    E = ex + 1023;
    fx_range(E, f, 0, L.fu, L.g, s, side ? 0 : 1);
    ok = E < FX_BAD;
    if (ok) fx_hops(acc, E, f, V, 0, L.fu, L.g, s, side ? 0 : 1, sp);
  }
  fx_exchange(acc);
  for (int i0 = 0; i0 < ntmax; i0 += RT) {
    __syncthreads();
    if (t < RT && i0 + t < nt) {
      RevTerm r;
      rev_term(L, B, src, side, j, slot, prev, i0 + t, r);
      r.k = fx_coef(kinv * r.c.re, kinv * r.c.im);
      terms[side][t] = r;
    }
    __syncthreads();
    const int n = min(RT, nt - i0);
    if (ok) fx_headroom(acc, E);
#pragma unroll 1
    for (int i = 0; i < n && ok; ++i) {
      const RevTerm& r = terms[side][i];
      zd p[6];
      fx_load_half(r.f, V, x, sp, p);
      ok = r.k.e != FX_BAD && fx_axpy_g5(acc, E, r.k, p);
    }
  }
  if (x >= V) return;
  zd a[6];
  if (ok) {
    const double ks = L.kappa * fx_pow2(E - FX_E_BIAS), us = fx_pow2(ex - 1079);
    zd h[6];
    fx_double(acc, h);
#pragma unroll
    for (int i = 0; i < 6; ++i) a[i] = us * fx_value(__ldg(f.c + (i < 3 ? sp * 3 + i : (2 + sp) * 3 + i - 3) * V + x));
    h_finish(a, h, mk(ks, 0.0));
  } else {
    Spinor<double> b;
    rev_site_fp64(L, B, src, side, j, slot, prev, nt, x, &b);
    fx_pick(b, sp, a);
  }
  fx_store_half((side ? B.gw_new : B.gv_new) + src * L.vs, V, x, sp, a);
}
void fx_rev_stencil(const Lat<double>& L, const Rev<double>& B, int j, int slot, int prev, int nrec,
                    cudaStream_t st) {
  const int64_t V = L.g.V;
  const int sx = V * L.nsrc < 152 * 32 ? 16 : 32;
  k_fx_rev<<<dim3(nblocks(V, sx), L.nsrc), 4 * sx, 0, st>>>(L, B, j, slot, prev, nrec);
}

}  // namespace ov
