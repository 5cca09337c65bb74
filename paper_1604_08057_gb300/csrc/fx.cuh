// FP64-accurate lattice arithmetic on the integer pipes.
//
// GB300 issues 2 FP64 fused multiply-adds per SM and clock but 64 integer
// 32 x 32 + 64 -> 64 multiply-adds (both measured), so a product of two FP64
// numbers formed as three integer multiply-adds costs a tenth of one DFMA.
// Operands are held in block fixed point: all components of one site's spinor
// (or of one link) share a power-of-two scale taken from the largest of them,
// and each is an integer of 57 (59) bits split at bit 30 into a signed high part
// and a balanced low part |l| <= 2^29:
//     x = (h 2^30 + l) 2^-s.
// A product keeps h h', h l' and l h'; the dropped l l' is at most 2^-58 of the
// largest product.  Sums of products are exact in 64 bits (bounds at each use),
// and the sum over hops is kept to 2^-57 of the largest term, so a site's result
// carries an error of some 2^-56 of the largest contribution to it, against
// 2^-53 per operation in FP64 arithmetic.  A site whose field or links lie
// outside the exponent windows below (infinities, NaN, magnitudes far from 1) is
// marked by its exponent word, and every sum that meets it is formed in FP64.
#pragma once
#include "dslash.cuh"
#include "kernels.h"

namespace ov {

// Biased exponents (the 11-bit field of an FP64 number): |x| < 2^(e - 1022).
constexpr int FX_F_MIN = 200, FX_F_MAX = 1062;    // fields: 2^-822 .. 2^40
constexpr int FX_U_MIN = 900, FX_U_MAX = 1080;    // links: 2^-122 .. 2^58
constexpr int FX_C_MIN = 100, FX_C_MAX = 1900;    // coefficients: 2^-922 .. 2^878
constexpr int FX_E_BIAS = 2100;                   // a sum's unit is 2^(E - FX_E_BIAS)
constexpr int FX_BAD = 0x7fff;                    // exponent word of what needs FP64

typedef long long fxll;

struct FxInt { int h, l; };                       // h 2^30 + l
struct FxZ { fxll re, im; };

__device__ __forceinline__ FxInt fx_split(fxll x) {
  FxInt r;
  r.h = (int)((x + (1ll << 29)) >> 30);
  r.l = (int)((unsigned)x - ((unsigned)r.h << 30));
  return r;
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
__device__ __forceinline__ unsigned fx_max_mag(const Spinor<double>& p) {
  unsigned m = 0u;
#pragma unroll
  for (int i = 0; i < 12; ++i) m = max(m, max(fx_mag(p.c[i].re), fx_mag(p.c[i].im)));
  return m;
}
// exponent word of a field value of magnitude word m (zero counts as the smallest)
__device__ __forceinline__ int fx_field_exp(unsigned m) {
  const int e = (int)(m >> 20);
  return m == 0u ? FX_F_MIN : e < FX_F_MIN || e > FX_F_MAX ? FX_BAD : e;
}

// one site of a fixed-point field (layout of an FP64 field, an int4 (re.h, re.l, im.h, im.l)
// per complex component); where the site is out of the window only its exponent word is
// written, and true is returned: the caller keeps the FP64 values
__device__ __forceinline__ bool fx_store(const FxField& f, int64_t V, int64_t s, const Spinor<double>& p) {
  const int e = fx_field_exp(fx_max_mag(p));
  f.e[s] = (short)e;
  if (e == FX_BAD) return true;
#pragma unroll
  for (int i = 0; i < 12; ++i) {
    const FxInt r = fx_split(fx_conv(p.c[i].re, e)), q = fx_split(fx_conv(p.c[i].im, e));
    f.c[i * V + s] = make_int4(r.h, r.l, q.h, q.l);
  }
  return false;
}
// the FP64 values of a component in units of 2^(e - 1079)
__device__ __forceinline__ zd fx_value(int4 q) {
  return mk((double)(((fxll)q.x << 30) + q.y), (double)(((fxll)q.z << 30) + q.w));
}
// a fixed-point field read as FP64, from its FP64 companion where a site is out of the window
struct FxLoad {
  FxField f;
  const double* d;
  int64_t Vf, off;
  __device__ __forceinline__ void operator()(int64_t s, Spinor<double>& o) const {
    const int e = f.e[off + s];
    if (e == FX_BAD) {
      load_spinor(d, Vf, off + s, o);
      return;
    }
    const double u = fx_pow2(e - 1079);
    for (int i = 0; i < 12; ++i) o.c[i] = u * fx_value(f.c[i * Vf + off + s]);
  }
};

// one real product a b into (hh, x): a b ~ hh 2^60 + x 2^30
__device__ __forceinline__ void fx_mac(fxll& hh, fxll& x, int ah, int al, int bh, int bl) {
  hh += (fxll)ah * bh;
  x += (fxll)ah * bl;
  x += (fxll)al * bh;
}

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

// *E = max(*E, exponent of every hop's term); a marked field or link gives at least FX_BAD
__device__ __forceinline__ void fx_range(int& E, const FxField& f, int off, const FxLinks& U, const Geom& g,
                                         const FxSite& s, int dagger) {
  const int V = (int)g.V;
#pragma unroll
  for (int hop = 0; hop < 8; ++hop) {
    const int n = s.neighbour(g, hop);
    E = max(E, (int)f.e[off + n] + (int)U.ex[fx_link_dir(hop, dagger) * V + ((hop & 1) ? n : s.x)]);
  }
}
// ---------------------------------------------------------------------------
// Hop sums.  Two threads of a warp (lanes l and l + 16) share a site: thread sp handles
// spin sp of every half spinor (spins (sp, 2 + sp) or (sp, 3 - sp) of the neighbour),
// and ends up with spins sp and 2 + sp of the sum.  One thread per site needs 168
// registers, and with 12 warps on an SM the latencies of the integer chains show
// (apply_H, 4 sources on 6x18^3: 82 us; measured stalls: fixed latency and loads).
//
// With h = u_sp + SGN tau phase d and g = U h (or U^dagger h), the upper spin gains g and
// the lower spin +-phase (g_fwd - g_bwd): phase = i for x and z, 1 for y and t; d and the
// lower spin are spin 1 - sp's for x and y.
// ---------------------------------------------------------------------------
struct FxHalf {
  FxZ up[3], lo[3], xc[3];   // spins sp and 2 + sp; xc: the partner's lower spin
};
__device__ __forceinline__ void fx_zero(FxHalf& a) {
#pragma unroll
  for (int i = 0; i < 3; ++i) a.up[i] = a.lo[i] = a.xc[i] = FxZ{0, 0};
}
// g = U h (SGN > 0) or U^dagger h of one hop, in units of 2^(E - FX_E_BIAS)
template <int SGN>
__device__ __forceinline__ void fx_hop(FxZ (&g)[3], int E, const FxField& f, int64_t Vf, int off, const FxLinks& U,
                                       int V, int n, int x, int nu, int dir, int sp, int tau) {
  const int ls = SGN > 0 ? x : n;
  const int d = min(E - (int)f.e[off + n] - (int)U.ex[dir * V + ls], 62);
  int4 h[3];
  {
    const int pd = nu < 2 ? 3 - sp : 2 + sp;
    const int4* qu = f.c + ((int64_t)sp * 3 * Vf + off + n);
    const int4* qd = f.c + ((int64_t)pd * 3 * Vf + off + n);
    const int t = SGN * tau;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int4 u = __ldg(qu + a * Vf), q = __ldg(qd + a * Vf);
      // |h.h| < 2^28, |h.l| < 2^30: the halves of the split add without carry
      h[a] = (nu & 1) ? make_int4(u.x + t * q.x, u.y + t * q.y, u.z + t * q.z, u.w + t * q.w)
                      : make_int4(u.x - t * q.z, u.y - t * q.w, u.z + t * q.x, u.w + t * q.y);
    }
  }
  const fxll half = (1ll << d) >> 1;
  const int4* lk = U.e + ((int64_t)dir * 9 * V + ls);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    // six real products each: |hh| < 6 2^57, |x| < 6 (2^59 + 2^57)
    fxll hr = half, xr = 1ll << 29, hi = half, xi = 1ll << 29;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int4 u = __ldg(lk + (int64_t)(SGN > 0 ? a * 3 + b : b * 3 + a) * V);
      fx_mac(hr, xr, u.x, u.y, h[b].x, h[b].y);
      fx_mac(hi, xi, u.x, u.y, h[b].z, h[b].w);
      if (SGN > 0) {
        fx_mac(hr, xr, u.z, u.w, -h[b].z, -h[b].w);
        fx_mac(hi, xi, u.z, u.w, h[b].x, h[b].y);
      } else {
        fx_mac(hr, xr, u.z, u.w, h[b].z, h[b].w);
        fx_mac(hi, xi, u.z, u.w, -h[b].x, -h[b].y);
      }
    }
    g[a] = FxZ{(hr + (xr >> 30)) >> d, (hi + (xi >> 30)) >> d};
  }
}
// acc += the eight hops of D_w of field f (sites off + s of a Vf-site field).  A product is
// below 2^57 units, so the 48 of eight hops stay below 2^62.6 (for sixteen hops the caller
// takes E one higher).  The loop is kept rolled: fully unrolled, the code outgrows the
// instruction cache and instruction fetch sets the pace (144 us per step pair at 14^4).
__device__ __forceinline__ void fx_hops(FxHalf& acc, int E, const FxField& f, int64_t Vf, int off, const FxLinks& U,
                                        const Geom& g, const FxSite& st, int dagger, int sp) {
  const int V = (int)g.V;
#pragma unroll 1
  for (int nu = 0; nu < 4; ++nu) {
    const int tau = nu == 0 ? -1 : nu == 3 ? 1 : 2 * sp - 1;
    FxZ a[3], b[3];
    fx_hop<1>(a, E, f, Vf, off, U, V, st.neighbour(g, 2 * nu), st.x, nu, fx_link_dir(2 * nu, dagger), sp, tau);
    fx_hop<-1>(b, E, f, Vf, off, U, V, st.neighbour(g, 2 * nu + 1), st.x, nu, fx_link_dir(2 * nu + 1, dagger), sp,
               tau);
    const fxll m = (nu == 1 && sp == 0) || (nu == 2 && sp == 1) ? -1 : 0;   // the lower spin's sign
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      acc.up[i].re += a[i].re + b[i].re;
      acc.up[i].im += a[i].im + b[i].im;
      const FxZ t{((a[i].re - b[i].re) ^ m) - m, ((a[i].im - b[i].im) ^ m) - m};
      const FxZ q = (nu & 1) ? t : FxZ{-t.im, t.re};
      if (nu < 2) {
        acc.xc[i].re += q.re;
        acc.xc[i].im += q.im;
      } else {
        acc.lo[i].re += q.re;
        acc.lo[i].im += q.im;
      }
    }
  }
}
// the partner's part of the lower spin (every lane of the warp)
__device__ __forceinline__ void fx_exchange(FxHalf& a) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    a.lo[i].re += __shfl_xor_sync(0xffffffffu, a.xc[i].re, 16);
    a.lo[i].im += __shfl_xor_sync(0xffffffffu, a.xc[i].im, 16);
  }
}

// ---------------------------------------------------------------------------
// sums of coefficient times field at one site (the thread's two spins)
// ---------------------------------------------------------------------------
struct FxCoef { int rh, rl, ih, il, e; };         // 59-bit complex coefficient and its exponent
__device__ __forceinline__ FxCoef fx_coef(double re, double im) {
  const unsigned m = max(fx_mag(re), fx_mag(im));
  const int ex = m == 0u ? 1022 : (int)(m >> 20);
  if (ex < FX_C_MIN || ex > FX_C_MAX) return FxCoef{0, 0, 0, 0, FX_BAD};
  const double f = fx_pow2(59 - (ex - 1022));
  const FxInt a = fx_split(__double2ll_rn(re * f)), b = fx_split(__double2ll_rn(im * f));
  return FxCoef{a.h, a.l, b.h, b.l, ex};
}
__device__ __forceinline__ void fx_shift(FxHalf& a, int& E, int sh) {
  const fxll r = (1ll << sh) >> 1;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    a.up[i].re = (a.up[i].re + r) >> sh;
    a.up[i].im = (a.up[i].im + r) >> sh;
    a.lo[i].re = (a.lo[i].re + r) >> sh;
    a.lo[i].im = (a.lo[i].im + r) >> sh;
  }
  E += sh;
}
__device__ __forceinline__ int fx_top(FxZ a) {
  const int x = (int)(a.re >> 32), y = (int)(a.im >> 32);
  return (x ^ (x >> 31)) | (y ^ (y >> 31));
}
// Room for 16 more terms (each below 2^57 units): a sum that may pass 2^60 is shifted down
// by two bits (rounded), which leaves it below 2^60.6.
__device__ __forceinline__ void fx_headroom(FxHalf& a, int& E) {
  int m = 0;
#pragma unroll
  for (int i = 0; i < 3; ++i) m |= fx_top(a.up[i]) | fx_top(a.lo[i]);
  if (m >= (1 << 28)) fx_shift(a, E, 2);
}
// one component of a 57-bit field times a coefficient, in units 2^d below the sum's
__device__ __forceinline__ FxZ fx_coef_mul(const FxCoef& c, zd p, int e, int d, fxll half) {
  const FxInt r = fx_split(fx_conv(p.re, e)), q = fx_split(fx_conv(p.im, e));
  fxll hr = half, xr = 1ll << 29, hi = half, xi = 1ll << 29;
  fx_mac(hr, xr, c.rh, c.rl, r.h, r.l);
  fx_mac(hr, xr, c.ih, c.il, -q.h, -q.l);
  fx_mac(hi, xi, c.rh, c.rl, q.h, q.l);
  fx_mac(hi, xi, c.ih, c.il, r.h, r.l);
  return FxZ{(hr + (xr >> 30)) >> d, (hi + (xi >> 30)) >> d};
}
// up -= c p, lo += c p (the pattern under which gamma5 (-kappa acc) gains kappa c p on both);
// p: the thread's six components; false when they are out of the window
__device__ __forceinline__ bool fx_axpy_g5(FxHalf& acc, int& E, const FxCoef& c, const zd (&p)[6]) {
  unsigned m = 0u;
#pragma unroll
  for (int i = 0; i < 6; ++i) m = max(m, max(fx_mag(p[i].re), fx_mag(p[i].im)));
  const int e = fx_field_exp(m);
  if (e == FX_BAD) return false;
  const int et = e + c.e;
  if (et > E) {
    fx_shift(acc, E, min(et - E, 62));
    E = et;   // (a shift of 62 leaves nothing of the old sum)
  }
  const int d = E - et;
  if (d > 59) return true;   // below half a unit
  const fxll half = (1ll << d) >> 1;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const FxZ u = fx_coef_mul(c, p[i], e, d, half), l = fx_coef_mul(c, p[3 + i], e, d, half);
    acc.up[i].re -= u.re;
    acc.up[i].im -= u.im;
    acc.lo[i].re += l.re;
    acc.lo[i].im += l.im;
  }
  return true;
}
// the thread's six components (spins sp and 2 + sp) of a site of an FP64 field
__device__ __forceinline__ void fx_load_half(const double* f, int64_t V, int64_t s, int sp, zd (&p)[6]) {
  const double2* q = reinterpret_cast<const double2*>(f) + s;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const double2 a = __ldg(q + (sp * 3 + i) * V), b = __ldg(q + ((2 + sp) * 3 + i) * V);
    p[i] = mk(a.x, a.y);
    p[3 + i] = mk(b.x, b.y);
  }
}
__device__ __forceinline__ void fx_store_half(double* f, int64_t V, int64_t s, int sp, const zd (&p)[6]) {
  double2* q = reinterpret_cast<double2*>(f) + s;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    q[(sp * 3 + i) * V] = make_double2(p[i].re, p[i].im);
    q[((2 + sp) * 3 + i) * V] = make_double2(p[3 + i].re, p[3 + i].im);
  }
}
// the same six of a full spinor
__device__ __forceinline__ void fx_pick(const Spinor<double>& t, int sp, zd (&p)[6]) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    p[i] = sp ? t.c[3 + i] : t.c[i];
    p[3 + i] = sp ? t.c[9 + i] : t.c[6 + i];
  }
}

}  // namespace ov
