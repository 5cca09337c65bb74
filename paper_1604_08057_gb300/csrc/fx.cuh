// Lattice sums of FP64 accuracy on the integer pipes, for the operator.
//
// GB300 issues 2 FP64 fused multiply-adds per SM and clock but 64 integer
// 32 x 32 + 64 -> 64 multiply-adds (both measured), so a product of two FP64
// numbers formed as three integer multiply-adds costs a tenth of one DFMA.
// The operator's input and links are held in block fixed point: the 24 reals of a
// site's spinor (the 18 of a link) share a power-of-two scale taken from the
// largest of them, and each is an integer of 57 (59) bits split at bit 30 into a
// signed high part and a balanced low part |l| <= 2^29:
//     x = (h 2^30 + l) 2^(e - 1079)        (links: 2^(e - 1081)),
// e being the largest component's biased FP64 exponent, |x| < 2^(e - 1022).  A
// component within 2^-4 of the site's largest keeps all of its FP64 bits; one 2^-n
// below it keeps 57 - n of them.
// A product keeps h h', h l' and l h'; the dropped l l' is at most 2^-58 of the
// largest product.  Sums of products are exact in 64 bits (bounds at each use),
// with their own scale E: units of 2^(E - 2100), kept to some 2^-56 of the largest
// contribution to the site, against 2^-53 per operation in FP64 arithmetic.
// Infinities, NaN and magnitudes outside the window below mark a site (FX_BAD), and
// every sum that meets a marked site or link, or whose terms may leave FP64's range, is
// formed in FP64.
//
// The Lanczos recurrence and its derivatives stay in FP64: see setup() in ov_api.cu.
#pragma once
#include "dslash.cuh"
#include "kernels.h"

namespace ov {

// Biased exponents (the 11-bit field of an FP64 number): |x| < 2^(e - 1022).
constexpr int FX_F_MIN = 200, FX_F_MAX = 1900;    // fields: 2^-822 .. 2^878
constexpr int FX_U_MIN = 100, FX_U_MAX = 1900;    // links: 2^-922 .. 2^878
constexpr int FX_E_BIAS = 2100;                   // a sum's unit is 2^(E - FX_E_BIAS)
constexpr int FX_BAD = 0x7fff;                    // exponent word of a marked site or link

typedef long long fxll;

struct FxInt { int h, l; };                       // h 2^30 + l
struct FxZ { fxll re, im; };

__device__ __forceinline__ FxInt fx_split(fxll x) {
  FxInt r;
  r.h = (int)((x + (1ll << 29)) >> 30);
  r.l = (int)((unsigned)x - ((unsigned)r.h << 30));
  return r;
}
__device__ __forceinline__ fxll fx_join(int h, int l) { return ((fxll)h << 30) + l; }
// 64-bit shifts by 0 <= n <= 31: two instructions (a shift by any n < 64 takes five)
__device__ __forceinline__ fxll fx_sar(fxll v, int n) {
  const int lo = (int)v, hi = (int)(v >> 32);
  return ((fxll)(hi >> n) << 32) | (unsigned)__funnelshift_r(lo, hi, n);
}
__device__ __forceinline__ unsigned fx_mag(double d) { return (unsigned)__double2hiint(d) & 0x7fffffffu; }
// 2^s as an FP64 number, |s| <= 1022
__device__ __forceinline__ double fx_pow2(int s) { return __hiloint2double((s + 1023) * (1 << 20), 0); }

// d 2^(1079 - e) to the nearest integer (|d| < 2^(e - 1022) gives 57 bits), in integer
// operations: a conversion instruction runs at the FP64 rate
__device__ __forceinline__ fxll fx_conv(double d, int e) {
  const int hi = __double2hiint(d);
  const int n = min(e - ((hi >> 20) & 0x7ff), 63);
  const unsigned long long m =
      ((unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 32 | (unsigned)__double2loint(d)) << 5;
  const fxll t = (fxll)(((m >> n) + 1ull) >> 1);
  return hi < 0 ? -t : t;
}
// exponent word of a field value of magnitude word m (zero counts as the smallest)
__device__ __forceinline__ int fx_field_exp(unsigned m) {
  const int e = (int)(m >> 20);
  return m == 0u ? FX_F_MIN : e < FX_F_MIN || e > FX_F_MAX ? FX_BAD : e;
}

// ---------------------------------------------------------------------------
// Fields.  Tiles of 32 sites: component c of site s is the int4 (re.h, re.l, im.h, im.l)
// at (s / 32) * 384 + c * 32 + s % 32, so every component of a site is at a constant
// offset from one address; exponents at e[s].
//
// Two threads of a warp (lanes l and l + 16) share a site: thread sp holds spins sp and
// 2 + sp (components 0..2 and 3..5 of its arrays).
// ---------------------------------------------------------------------------
__device__ __forceinline__ int64_t fx_at(int64_t s) { return (s >> 5) * 384 + (s & 31); }
// thread t of a group of 2 n threads: site t / 32 * 16 + t % 16, spin (t / 16) % 2
__device__ __forceinline__ int fx_site_of(int t) { return (t >> 5) * 16 + (t & 15); }
__device__ __forceinline__ int fx_spin_of(int t) { return (t >> 4) & 1; }
__device__ __forceinline__ int fx_comp(int sp, int i) { return i < 3 ? sp * 3 + i : 3 + sp * 3 + i; }

struct FxH {
  int4 q[6];
  int e;
};
__device__ __forceinline__ void fx_put(const FxField& f, int64_t s, int sp, const FxH& o) {
  int4* p = f.c + fx_at(s) + sp * 96;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    p[i * 32] = o.q[i];
    p[192 + i * 32] = o.q[3 + i];
  }
  if (sp == 0) f.e[s] = (short)o.e;
}
// a site of a fixed-point field read as FP64, from its FP64 companion (site-major, V sites)
// where the site is marked
struct FxLoad {
  FxField f;
  const double* d;
  int64_t V;
  __device__ __forceinline__ void operator()(int64_t s, Spinor<double>& o) const {
    const int e = f.e[s];
    if (e == FX_BAD) return load_spinor(d, V, s, o);
    const double u = fx_pow2(e - 1079);
    const int4* p = f.c + fx_at(s);
    for (int i = 0; i < 12; ++i) {
      const int4 q = p[i * 32];
      o.c[i] = mk(u * (double)fx_join(q.x, q.y), u * (double)fx_join(q.z, q.w));
    }
  }
};

// acc += a b as one multiply-add (written out, so that sums are not re-associated into
// products and separate 64-bit additions)
__device__ __forceinline__ void fx_wide(fxll& acc, int a, int b) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}
// one real product a b into (hh, x): a b ~ hh 2^60 + x 2^30
__device__ __forceinline__ void fx_mac(fxll& hh, fxll& x, int ah, int al, int bh, int bl) {
  fx_wide(hh, ah, bh);
  fx_wide(x, ah, bl);
  fx_wide(x, al, bh);
}
// acc += a b, acc += conj(a) b (acc as hh and x sums of its two parts)
struct FxAcc { fxll hr, xr, hi, xi; };
__device__ __forceinline__ void fx_cmac(FxAcc& c, int4 a, int4 b) {
  fx_mac(c.hr, c.xr, a.x, a.y, b.x, b.y);
  fx_mac(c.hr, c.xr, a.z, a.w, -b.z, -b.w);
  fx_mac(c.hi, c.xi, a.x, a.y, b.z, b.w);
  fx_mac(c.hi, c.xi, a.z, a.w, b.x, b.y);
}
__device__ __forceinline__ void fx_cdot(FxAcc& c, int4 a, int4 b) {
  fx_mac(c.hr, c.xr, a.x, a.y, b.x, b.y);
  fx_mac(c.hr, c.xr, a.z, a.w, b.z, b.w);
  fx_mac(c.hi, c.xi, a.x, a.y, b.z, b.w);
  fx_mac(c.hi, c.xi, a.z, a.w, -b.x, -b.y);
}

// ---------------------------------------------------------------------------
// a thread's six components of a sum, in units of 2^(E - FX_E_BIAS)
// ---------------------------------------------------------------------------
struct FxHalf {
  FxZ v[6];
  int E;
};
__device__ __forceinline__ void fx_zero(FxHalf& a, int E) {
#pragma unroll
  for (int i = 0; i < 6; ++i) a.v[i] = FxZ{0, 0};
  a.E = E;
}
// whether a sum's unit is a normal FP64 number (E includes FX_BAD's)
__device__ __forceinline__ bool fx_scale_ok(int E) { return E >= FX_E_BIAS - 1022 && E <= FX_E_BIAS + 1023; }
// the sum's FP64 values
__device__ __forceinline__ void fx_double(const FxHalf& a, zd (&o)[6]) {
  const double u = fx_pow2(a.E - FX_E_BIAS);
#pragma unroll
  for (int i = 0; i < 6; ++i) o[i] = mk(u * (double)a.v[i].re, u * (double)a.v[i].im);
}
// six FP64 components encoded (every lane)
__device__ __forceinline__ void fx_from_double(const zd (&p)[6], FxH& o) {
  unsigned m = 0u;
#pragma unroll
  for (int i = 0; i < 6; ++i) m = max(m, max(fx_mag(p[i].re), fx_mag(p[i].im)));
  m = max(m, __shfl_xor_sync(0xffffffffu, m, 16));
  const int e = fx_field_exp(m);
  o.e = e;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const FxInt x = fx_split(fx_conv(p[i].re, e == FX_BAD ? 2100 : e)), y = fx_split(fx_conv(p[i].im, e == FX_BAD ? 2100 : e));
    o.q[i] = make_int4(x.h, x.l, y.h, y.l);
  }
}

// ---------------------------------------------------------------------------
// hop sums
// ---------------------------------------------------------------------------
// Links: five "directions" x, y, z, e^{mu} t, e^{-mu} t; entry q of direction d of site s at
// (s / 32) * 1440 + (d * 9 + q) * 32 + s % 32, its exponent at ex[d * V + s].
__device__ __forceinline__ int64_t fx_link_at(int64_t s, int d) { return (s >> 5) * 1440 + d * 288 + (s & 31); }

// Site x and its coordinates; hop 0..7 is direction hop / 2, forward for even hop.
struct FxSite {
  int x, c0, c1, c2, c3;
  __device__ __forceinline__ FxSite(const Geom& g, int64_t s) {
    int c[4];
    site_coords(g, s, c);
    x = (int)s;
    c0 = c[0]; c1 = c[1]; c2 = c[2]; c3 = c[3];
  }
  __device__ __forceinline__ int neighbour(const Geom& g, int hop) const {
    const int nu = hop >> 1;
    const int c = nu == 0 ? c0 : nu == 1 ? c1 : nu == 2 ? c2 : c3;
    const int n = nu == 0 ? g.nx : nu == 1 ? g.ny : nu == 2 ? g.nz : g.nt;
    const int st = nu == 0 ? 1 : nu == 1 ? g.nx : nu == 2 ? g.nx * g.ny : g.nx * g.ny * g.nz;
    if (hop & 1) return c == 0 ? x + (n - 1) * st : x - st;
    return c == n - 1 ? x - (n - 1) * st : x + st;
  }
};
// link "direction" of a hop: H uses e^{mu} forward and e^{-mu} backward in t, H^dagger the reverse
__device__ __forceinline__ int fx_link_dir(int hop, int dagger) { return hop < 6 ? hop >> 1 : 3 + ((hop & 1) ^ dagger); }

// exponents of the eight hops' terms, 16 bits each: forward hops in f, backward in b
struct FxExps {
  unsigned long long f, b;
};
// the largest exponent of the hops' terms; a marked field or link gives at least FX_BAD
__device__ __forceinline__ int fx_range(FxExps& x, const FxField& f, const FxLinks& U, const Geom& g, const FxSite& s,
                                        int dagger) {
  const int V = (int)g.V;
  int E = 0;
  x.f = x.b = 0ull;
#pragma unroll
  for (int hop = 0; hop < 8; ++hop) {
    const int n = s.neighbour(g, hop);
    const int e = (int)f.e[n] + (int)U.ex[fx_link_dir(hop, dagger) * V + ((hop & 1) ? n : s.x)];
    E = max(E, e);
    if (hop & 1) x.b |= (unsigned long long)(unsigned)e << (hop >> 1) * 16;
    else x.f |= (unsigned long long)(unsigned)e << (hop >> 1) * 16;
  }
  return E;
}
// Thread sp handles spin sp of every half spinor: with h = u_sp + SGN tau phase d and g = U h
// (U^dagger h backward), the upper spin gains g and the lower spin +-phase (g_fwd - g_bwd);
// phase = i for x and z, 1 for y and t; d and that lower spin are the partner's for x and y.
// g is in units of 2^(E - FX_E_BIAS).
// The neighbour's six int4 and the link's nine come through shared memory, copied
// asynchronously one hop ahead: with the loads in registers a warp waits for each hop's
// data, and 16 warps on an SM do not cover that (H and H^dagger at 14^4: 67 us so; stalls on
// loads 5.7 cycles out of 11).
// One such area per warp: everything in it is written and read by that warp's lanes.
union FxStage {
  struct {
    int4 q[2][6][32];            // [hop parity][component][lane]
    int4 u[2][9][16];            // [hop parity][entry][site]
    int nb[8][16];               // neighbours of the hops
  };
  double2 out[16 * 13];          // rows of the user's layout
};
__device__ __forceinline__ void fx_copy16(int4* dst, const int4* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void fx_copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void fx_copy_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void fx_hop_copy(FxStage& S, const FxField& f, const FxLinks& U, int x, int hop,
                                            int dagger, int sp) {
  if (hop < 8) {
    const int p = hop & 1, t = threadIdx.x & 31, n = S.nb[hop][t & 15];
    const int4* q = f.c + fx_at(n);
    const int4* qu = q + sp * 96;
    const int4* qd = q + (hop < 4 ? 3 - sp : 2 + sp) * 96;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      fx_copy16(&S.q[p][a][t], qu + a * 32);
      fx_copy16(&S.q[p][3 + a][t], qd + a * 32);
    }
    const int4* lk = U.e + fx_link_at(p ? n : x, fx_link_dir(hop, dagger)) + sp * 160;
#pragma unroll
    for (int i = 0; i < 5; ++i)
      if (sp == 0 || i < 4) fx_copy16(&S.u[p][sp * 5 + i][t & 15], lk + i * 32);
  }
  fx_copy_commit();   // an empty group past the last hop keeps the waits' counts
}
template <int SGN>
__device__ __forceinline__ void fx_hop(FxZ (&g)[3], const FxStage& S, int d, int nu, int sp, int tau) {
  const int t = threadIdx.x & 31, slot = t & 15, p = SGN > 0 ? 0 : 1;
  int4 h[3];
  const int s = SGN * tau;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int4 u = S.q[p][a][t], w = S.q[p][3 + a][t];
    // |h.h| < 2^28, |h.l| < 2^30: the halves of the split add without carry
    h[a] = (nu & 1) ? make_int4(u.x + s * w.x, u.y + s * w.y, u.z + s * w.z, u.w + s * w.w)
                    : make_int4(u.x - s * w.z, u.y - s * w.w, u.z + s * w.x, u.w + s * w.y);
  }
  const fxll half = (1ll << d) >> 1;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    // six real products each: |hh| < 6 2^57, |x| < 6 (2^59 + 2^57)
    FxAcc c{half, 1ll << 29, half, 1ll << 29};
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int4 u = S.u[p][SGN > 0 ? a * 3 + b : b * 3 + a][slot];
      if (SGN > 0) fx_cmac(c, u, h[b]);
      else fx_cdot(c, u, h[b]);
    }
    g[a] = FxZ{fx_sar(c.hr + (c.xr >> 30), min(d, 31)), fx_sar(c.hi + (c.xi >> 30), min(d, 31))};
  }
  if (d > 31) {
#pragma unroll
    for (int a = 0; a < 3; ++a) g[a] = FxZ{g[a].re >> (d - 31), g[a].im >> (d - 31)};
  }
}
__device__ __forceinline__ void fx_swap_lower(FxHalf& a) {
#pragma unroll
  for (int i = 3; i < 6; ++i) {
    a.v[i].re = __shfl_xor_sync(0xffffffffu, a.v[i].re, 16);
    a.v[i].im = __shfl_xor_sync(0xffffffffu, a.v[i].im, 16);
  }
}
// acc += the hops of D_w of field f at acc's scale; every lane of the warp.  A product is below
// 2^57 units, so the 48 of eight hops stay below 2^62.6.  The loop is kept rolled: fully
// unrolled, the code outgrows the instruction cache and instruction fetch sets the pace (H and
// H^dagger at 14^4: 144 us so, 71 rolled).  Copies in flight and the data read belong to one warp.
__device__ __forceinline__ void fx_hops(FxHalf& acc, const FxField& f, const FxLinks& U, const Geom& g,
                                        const FxSite& st, const FxExps& ex, int dagger, int sp, FxStage& S) {
  __syncwarp();
  if (sp == 0) {
#pragma unroll
    for (int hop = 0; hop < 8; ++hop) S.nb[hop][threadIdx.x & 15] = st.neighbour(g, hop);
  }
  __syncwarp();
  fx_hop_copy(S, f, U, st.x, 0, dagger, sp);
  fx_hop_copy(S, f, U, st.x, 1, dagger, sp);
  fx_swap_lower(acc);   // x and y feed the partner's lower spin
#pragma unroll 1
  for (int nu = 0; nu < 4; ++nu) {
    const int tau = nu == 0 ? -1 : nu == 3 ? 1 : 2 * sp - 1;
    if (nu == 2) fx_swap_lower(acc);
    FxZ a[3], b[3];
    fx_copy_wait<1>();
    __syncwarp();
    fx_hop<1>(a, S, max(0, min(acc.E - (int)((ex.f >> (16 * nu)) & 0xffff), 62)), nu, sp, tau);
    __syncwarp();
    fx_hop_copy(S, f, U, st.x, 2 * nu + 2, dagger, sp);
    fx_copy_wait<1>();
    __syncwarp();
    fx_hop<-1>(b, S, max(0, min(acc.E - (int)((ex.b >> (16 * nu)) & 0xffff), 62)), nu, sp, tau);
    __syncwarp();
    fx_hop_copy(S, f, U, st.x, 2 * nu + 3, dagger, sp);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      acc.v[i].re += a[i].re + b[i].re;
      acc.v[i].im += a[i].im + b[i].im;
      a[i].re -= b[i].re;
      a[i].im -= b[i].im;
    }
    if (nu == 1 || nu == 2) {   // the lower spin's sign: - for (y, spin 0) and (z, spin 1)
      const fxll m = (nu == 1) == (sp == 0) ? -1 : 0;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        a[i].re = (a[i].re ^ m) - m;
        a[i].im = (a[i].im ^ m) - m;
      }
    }
    if (nu & 1) {
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        acc.v[3 + i].re += a[i].re;
        acc.v[3 + i].im += a[i].im;
      }
    } else {
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        acc.v[3 + i].re -= a[i].im;
        acc.v[3 + i].im += a[i].re;
      }
    }
  }
  fx_copy_wait<0>();
}

}  // namespace ov
