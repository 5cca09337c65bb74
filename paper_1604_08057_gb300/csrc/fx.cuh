// FP64-accurate lattice arithmetic on the integer pipes.
//
// GB300 issues 2 FP64 fused multiply-adds per SM and clock but 64 integer
// 32 x 32 + 64 -> 64 multiply-adds (both measured), so a product of two FP64
// numbers formed as three integer multiply-adds costs a tenth of one DFMA.
// Every field of an FP64 call is held in block fixed point: the 24 reals of a
// site's spinor (the 18 of a link) share a power-of-two scale taken from the
// largest of them, and each is an integer of 57 (59) bits split at bit 30 into a
// signed high part and a balanced low part |l| <= 2^29:
//     x = (h 2^30 + l) 2^(e - 1079)        (links: 2^(e - 1081)),
// e being the largest component's biased FP64 exponent, |x| < 2^(e - 1022).  A
// component within 2^-4 of the site's largest keeps more bits than FP64 has.
// A product keeps h h', h l' and l h'; the dropped l l' is at most 2^-58 of the
// largest product.  Sums of products are exact in 64 bits (bounds at each use),
// with their own scale E: units of 2^(E - 2100), kept to some 2^-56 of the largest
// contribution to the site, against 2^-53 per operation in FP64 arithmetic.
// Infinities, NaN and magnitudes outside the window below mark a site (FX_BAD);
// the operator's own entry points then use FP64 for every sum that meets it.  In
// the Lanczos recurrence a site (or link) below the window is zero, and a marked
// one is what a NaN is in FP64: it reaches the next dot product and stops the
// source with a non-finite error (above the window the norm overflows in FP64 too).
#pragma once
#include "dslash.cuh"
#include "kernels.h"

namespace ov {

// Biased exponents (the 11-bit field of an FP64 number): |x| < 2^(e - 1022).
constexpr int FX_F_MIN = 200, FX_F_MAX = 1900;    // fields: 2^-822 .. 2^878
constexpr int FX_U_MIN = 100, FX_U_MAX = 1900;    // links: 2^-922 .. 2^878
constexpr int FX_C_MIN = 100, FX_C_MAX = 1900;    // coefficients: 2^-922 .. 2^878
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
__device__ __forceinline__ fxll fx_shl(fxll v, int n) {
  const int lo = (int)v, hi = (int)(v >> 32);
  return ((fxll)(int)__funnelshift_l(lo, hi, n) << 32) | ((unsigned)lo << n);
}
__device__ __forceinline__ unsigned fx_mag(double d) { return (unsigned)__double2hiint(d) & 0x7fffffffu; }
// 2^s as an FP64 number, |s| <= 1022
__device__ __forceinline__ double fx_pow2(int s) { return __hiloint2double((s + 1023) * (1 << 20), 0); }
// 2^s for any s an exponent sum can give (0 or infinity past the FP64 range)
__device__ __forceinline__ double fx_pow2_wide(int s) {
  return s < -1022 ? 0.0 : s > 1023 ? __longlong_as_double(0x7ff0000000000000ll) : fx_pow2(s);
}
__device__ __forceinline__ double fx_nan() { return __longlong_as_double(0x7ff8000000000000ll); }

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
__device__ __forceinline__ void fx_load(const FxField& f, int64_t s, int sp, FxH& o) {
  const int4* p = f.c + fx_at(s) + sp * 96;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    o.q[i] = p[i * 32];
    o.q[3 + i] = p[192 + i * 32];
  }
  o.e = f.e[s];
}
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
  int64_t Vf, off;
  __device__ __forceinline__ void operator()(int64_t s, Spinor<double>& o) const {
    const int e = f.e[off + s];
    if (e == FX_BAD) {
      if (d) {
        load_spinor(d, Vf, off + s, o);
      } else {
        for (int i = 0; i < 12; ++i) o.c[i] = mk(fx_nan(), fx_nan());
      }
      return;
    }
    const double u = fx_pow2(e - 1079);
    const int4* p = f.c + fx_at(off + s);
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
__device__ __forceinline__ void fx_shift(FxHalf& a, int sh) {
  const fxll r = (1ll << sh) >> 1;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    a.v[i].re = (a.v[i].re + r) >> sh;
    a.v[i].im = (a.v[i].im + r) >> sh;
  }
  a.E += sh;
}
// make room for a term of exponent e (|term| < 2^57 units after it)
__device__ __forceinline__ void fx_raise(FxHalf& a, int e) {
  if (e > a.E) {
    fx_shift(a, min(e - a.E, 62));
    a.E = e;   // (a shift of 62 leaves nothing of the old sum)
  }
}
__device__ __forceinline__ int fx_top(FxZ a) {
  const int x = (int)(a.re >> 32), y = (int)(a.im >> 32);
  return (x ^ (x >> 31)) | (y ^ (y >> 31));
}
// Encode the sum: 57 bits below its largest component (of the site's two threads: every lane
// of the warp).  bad marks the site; a site below 2^(zero_top - FX_E_BIAS) becomes zero.
__device__ __forceinline__ void fx_encode(const FxHalf& a, bool bad, FxH& o, int zero_top = 0) {
  unsigned long long m = 0ull;
#pragma unroll
  for (int i = 0; i < 6; ++i)
    m |= (unsigned long long)(a.v[i].re ^ (a.v[i].re >> 63)) | (unsigned long long)(a.v[i].im ^ (a.v[i].im >> 63));
  // the two threads' scales may differ: bring the smaller bit count up to the larger scale
  const int bits = m ? 64 - __clzll((long long)m) : 0;      // |v| <= 2^bits
  int top = m ? a.E + bits : 0;                             // |v| <= 2^(top - FX_E_BIAS)
  top = max(top, __shfl_xor_sync(0xffffffffu, top, 16));
  const bool any = __shfl_xor_sync(0xffffffffu, (int)bad, 16) || bad;
  int e = top - 1078;                                       // |v| <= 2^(e - 1022)
  if (any || e > FX_F_MAX) e = FX_BAD;
  const bool none = top <= zero_top || e < FX_F_MIN;
  if (none && e != FX_BAD) e = FX_F_MIN;
  o.e = e;
  // to units of 2^(e - 1079) = 2^(top - 57 - FX_E_BIAS): down by r bits (rounded) or up by -r;
  // a sum of several terms has r = 0 .. 6
  const int r = top - 57 - a.E;
  if (!none && r >= 0 && r < 32) {
    const fxll h = (1ll << r) >> 1;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      const FxInt x = fx_split(fx_sar(a.v[i].re + h, r)), y = fx_split(fx_sar(a.v[i].im + h, r));
      o.q[i] = make_int4(x.h, x.l, y.h, y.l);
    }
  } else {
    const bool zero = none || r >= 62;
    const int up = min(max(-r, 0), 62), dn = min(max(r, 0), 62);
    const fxll h = (1ll << dn) >> 1;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      const FxInt x = fx_split(zero ? 0 : ((a.v[i].re << up) + h) >> dn);
      const FxInt y = fx_split(zero ? 0 : ((a.v[i].im << up) + h) >> dn);
      o.q[i] = make_int4(x.h, x.l, y.h, y.l);
    }
  }
}
// the sum's FP64 values
__device__ __forceinline__ void fx_double(const FxHalf& a, bool bad, zd (&o)[6]) {
  const double u = bad ? fx_nan() : fx_pow2_wide(a.E - FX_E_BIAS);
#pragma unroll
  for (int i = 0; i < 6; ++i) o[i] = mk(u * (double)a.v[i].re, u * (double)a.v[i].im);
}
// six FP64 components encoded (every lane); flush: a site below the window is encoded with the
// window's smallest exponent, to zero or to the bits above 2^-880, instead of marked
__device__ __forceinline__ void fx_from_double(const zd (&p)[6], FxH& o, bool flush = false) {
  unsigned m = 0u;
#pragma unroll
  for (int i = 0; i < 6; ++i) m = max(m, max(fx_mag(p[i].re), fx_mag(p[i].im)));
  m = max(m, __shfl_xor_sync(0xffffffffu, m, 16));
  const int e = flush && (int)(m >> 20) < FX_F_MIN ? FX_F_MIN : fx_field_exp(m);
  o.e = e;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const FxInt x = fx_split(fx_conv(p[i].re, e == FX_BAD ? 2100 : e)), y = fx_split(fx_conv(p[i].im, e == FX_BAD ? 2100 : e));
    o.q[i] = make_int4(x.h, x.l, y.h, y.l);
  }
}

// ---------------------------------------------------------------------------
// coefficients
// ---------------------------------------------------------------------------
struct FxCoef {
  int4 c;        // 59 bits: (re.h, re.l, im.h, im.l), c 2^(e - 1081)
  int e;
};
__device__ __forceinline__ FxCoef fx_coef(zd z) {
  const unsigned m = max(fx_mag(z.re), fx_mag(z.im));
  const int ex = m == 0u ? FX_C_MIN : (int)(m >> 20);
  FxCoef r{make_int4(0, 0, 0, 0), ex};
  if (ex < FX_C_MIN || ex > FX_C_MAX) {
    if (ex > FX_C_MAX) r.e = FX_BAD;   // (a smaller one is a zero)
    else r.e = FX_C_MIN;
    return r;
  }
  // 59 bits = 4 times the 57-bit conversion (an FP64 number has 53)
  const FxInt a = fx_split(4 * fx_conv(z.re, ex)), b = fx_split(4 * fx_conv(z.im, ex));
  r.c = make_int4(a.h, a.l, b.h, b.l);
  return r;
}
// acc += c f; false when f or c is marked
__device__ __forceinline__ bool fx_axpy(FxHalf& acc, const FxCoef& c, const FxH& f) {
  if (f.e == FX_BAD || c.e == FX_BAD) return false;
  const int et = f.e + c.e;
  fx_raise(acc, et);
  const int d = acc.E - et;
  if (d > 59) return true;   // below half a unit
  const fxll half = (1ll << d) >> 1;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    FxAcc t{half, 1ll << 29, half, 1ll << 29};
    fx_cmac(t, c.c, f.q[i]);
    fxll re = fx_sar(t.hr + (t.xr >> 30), min(d, 31)), im = fx_sar(t.hi + (t.xi >> 30), min(d, 31));
    if (d > 31) {
      re >>= d - 31;
      im >>= d - 31;
    }
    acc.v[i].re += re;
    acc.v[i].im += im;
  }
  return true;
}
// acc += f
__device__ __forceinline__ bool fx_add(FxHalf& acc, const FxH& f) {
  if (f.e == FX_BAD) return false;
  fx_raise(acc, f.e + 1021);                // f's integers are units of 2^(f.e + 1021 - FX_E_BIAS)
  const int d = acc.E - (f.e + 1021);
  if (d > 59) return true;
  const fxll half = (1ll << d) >> 1;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    fxll re = fx_sar(fx_join(f.q[i].x, f.q[i].y) + half, min(d, 31));
    fxll im = fx_sar(fx_join(f.q[i].z, f.q[i].w) + half, min(d, 31));
    if (d > 31) {
      re >>= d - 31;
      im >>= d - 31;
    }
    acc.v[i].re += re;
    acc.v[i].im += im;
  }
  return true;
}
// conj(a) b of a thread's six components as FP64: products of 57-bit fields, twelve per
// part: |hh| < 12 2^54, |x| < 12 2^57
__device__ __forceinline__ zd fx_dot(const FxH& a, const FxH& b) {
  FxAcc t{0, 0, 0, 0};
#pragma unroll
  for (int i = 0; i < 6; ++i) fx_cdot(t, a.q[i], b.q[i]);
  const double u = a.e == FX_BAD || b.e == FX_BAD ? fx_nan() : fx_pow2_wide(a.e + b.e - 2158 + 56);
  return mk(u * (double)((t.hr << 4) + (t.xr >> 26)), u * (double)((t.hi << 4) + (t.xi >> 26)));
}
// |a|^2 of a thread's six components
__device__ __forceinline__ double fx_norm2(const FxH& a) {
  fxll h = 0, x = 0;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    h += (fxll)a.q[i].x * a.q[i].x;
    h += (fxll)a.q[i].z * a.q[i].z;
    x += (fxll)a.q[i].x * a.q[i].y;
    x += (fxll)a.q[i].z * a.q[i].w;
  }
  const double u = a.e == FX_BAD ? fx_nan() : fx_pow2_wide(2 * a.e - 2158 + 56);
  return u * (double)((h << 4) + (x >> 25));
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
__device__ __forceinline__ int fx_range(FxExps& x, const FxField& f, int off, const FxLinks& U, const Geom& g,
                                        const FxSite& s, int dagger) {
  const int V = (int)g.V;
  int E = 0;
  x.f = x.b = 0ull;
#pragma unroll
  for (int hop = 0; hop < 8; ++hop) {
    const int n = s.neighbour(g, hop);
    const int e = (int)f.e[off + n] + (int)U.ex[fx_link_dir(hop, dagger) * V + ((hop & 1) ? n : s.x)];
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
// data, and 16 warps on an SM do not cover that (67 us per step pair at 14^4; stalls on
// loads 5.7 cycles out of 11).
// One such area per warp: everything in it is written and read by that warp's lanes.
struct FxRow {         // a thread's components of one field, handed to another thread
  int4 q[6][32];
  int e[32];
};
struct FxSumRow {      // a thread's components of a sum
  fxll v[12][32];
  int e[32];
};
constexpr int FX_RING = 3;
union FxStage {
  struct {
    int4 q[2][6][32];            // [hop parity][component][lane]
    int4 u[2][9][16];            // [hop parity][entry][site]
    int nb[8][16];               // neighbours of the hops
  };
  int4 ring[FX_RING][6][32];     // FxStream
  FxRow row;
  FxSumRow sum;
  double2 out[16 * 13];          // rows of the user's layout
};
__device__ __forceinline__ void fx_row_put(FxRow& r, const FxH& f) {
  const int t = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < 6; ++i) r.q[i][t] = f.q[i];
  r.e[t] = f.e;
}
__device__ __forceinline__ void fx_row_get(const FxRow& r, FxH& f) {
  const int t = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < 6; ++i) f.q[i] = r.q[i][t];
  f.e = r.e[t];
}
__device__ __forceinline__ void fx_copy16(int4* dst, const int4* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void fx_copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void fx_copy_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void fx_hop_copy(FxStage& S, const FxField& f, int off, const FxLinks& U, int x, int hop,
                                            int end, int dagger, int sp) {
  if (hop < end) {
    const int p = hop & 1, t = threadIdx.x & 31, n = S.nb[hop][t & 15];
    const int4* q = f.c + fx_at(off + n);
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
// acc += the hops of D_w of field f (sites off + s) in directions nu0 .. nu1 - 1 (all eight by
// default), at acc's scale; every lane of the warp.  A product is below 2^57 units, so the 48
// of eight hops stay below 2^62.6.  The loop
// is kept rolled: fully unrolled, the code outgrows the instruction cache and instruction fetch sets the pace (144 us per
// step pair at 14^4).  Copies in flight and the data read belong to one warp.
__device__ __forceinline__ void fx_hops(FxHalf& acc, const FxField& f, int off, const FxLinks& U, const Geom& g,
                                        const FxSite& st, const FxExps& ex, int dagger, int sp, FxStage& S,
                                        int nu0 = 0, int nu1 = 4) {
  __syncwarp();
  if (sp == 0) {
#pragma unroll
    for (int hop = 0; hop < 8; ++hop) S.nb[hop][threadIdx.x & 15] = st.neighbour(g, hop);
  }
  __syncwarp();
  fx_hop_copy(S, f, off, U, st.x, 2 * nu0, 2 * nu1, dagger, sp);
  fx_hop_copy(S, f, off, U, st.x, 2 * nu0 + 1, 2 * nu1, dagger, sp);
  if (nu0 < 2) fx_swap_lower(acc);   // x and y feed the partner's lower spin
#pragma unroll 1
  for (int nu = nu0; nu < nu1; ++nu) {
    const int tau = nu == 0 ? -1 : nu == 3 ? 1 : 2 * sp - 1;
    if (nu == 2 && nu0 < 2) fx_swap_lower(acc);
    FxZ a[3], b[3];
    fx_copy_wait<1>();
    __syncwarp();
    fx_hop<1>(a, S, max(0, min(acc.E - (int)((ex.f >> (16 * nu)) & 0xffff), 62)), nu, sp, tau);
    __syncwarp();
    fx_hop_copy(S, f, off, U, st.x, 2 * nu + 2, 2 * nu1, dagger, sp);
    fx_copy_wait<1>();
    __syncwarp();
    fx_hop<-1>(b, S, max(0, min(acc.E - (int)((ex.b >> (16 * nu)) & 0xffff), 62)), nu, sp, tau);
    __syncwarp();
    fx_hop_copy(S, f, off, U, st.x, 2 * nu + 3, 2 * nu1, dagger, sp);
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
  if (nu0 < 2 && nu1 <= 2) fx_swap_lower(acc);
}

// The sum of the partial sums that n warps formed for the same sites, in the first of them
// (n <= 4, each below 2^61.5 units of its own scale; EXACT: all of one scale and their sum
// below 2^63, as where the warps share the hops of one sum).  st[0 .. n - 1] are the warps'
// stages, w this warp's place.  Every thread of the block.
template <bool EXACT>
__device__ __forceinline__ void fx_join_warps(FxHalf& a, FxStage* st, int w, int n) {
  const int t = threadIdx.x & 31;
  __syncthreads();
  if (w > 0) {
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      st[w].sum.v[2 * i][t] = a.v[i].re;
      st[w].sum.v[2 * i + 1][t] = a.v[i].im;
    }
    st[w].sum.e[t] = a.E;
  }
  __syncthreads();
  if (w > 0) return;
  if (!EXACT) {
    int E = a.E;
    for (int k = 1; k < n; ++k) E = max(E, st[k].sum.e[t]);
    fx_shift(a, min(E + 2 - a.E, 62));
    a.E = E + 2;
  }
  for (int k = 1; k < n; ++k) {
    const int sh = min(a.E - st[k].sum.e[t], 62);
    const fxll r = (1ll << sh) >> 1;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      a.v[i].re += (st[k].sum.v[2 * i][t] + r) >> sh;
      a.v[i].im += (st[k].sum.v[2 * i + 1][t] + r) >> sh;
    }
  }
}

// A thread's components of a sequence of fields at one site, copied FX_RING - 1 vectors ahead
// (integers through shared memory, exponents in registers).  at(i): the i-th field.
// Every lane of the warp calls next() for i = 0, 1, .. n - 1.
struct FxStream {
  int e[FX_RING];
  template <typename At>
  __device__ __forceinline__ void issue(FxStage& S, int slot, int i, int n, int64_t s, int sp, const At& at) {
    if (i < n) {
      const FxField f = at(i);
      const int4* p = f.c + fx_at(s) + sp * 96;
      const int t = threadIdx.x & 31;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        fx_copy16(&S.ring[slot][a][t], p + a * 32);
        fx_copy16(&S.ring[slot][3 + a][t], p + 192 + a * 32);
      }
      e[slot] = f.e[s];
    }
    fx_copy_commit();
  }
  template <typename At>
  __device__ __forceinline__ void start(FxStage& S, int n, int64_t s, int sp, const At& at) {
#pragma unroll
    for (int i = 0; i < FX_RING - 1; ++i) issue(S, i, i, n, s, sp, at);
  }
  // field i of n into o, slot = i % FX_RING (a constant after unrolling)
  template <typename At>
  __device__ __forceinline__ void next(FxStage& S, int slot, int i, int n, int64_t s, int sp, const At& at, FxH& o) {
    issue(S, (slot + FX_RING - 1) % FX_RING, i + FX_RING - 1, n, s, sp, at);
    fx_copy_wait<FX_RING - 1>();
    const int t = threadIdx.x & 31;   // each thread reads its own copies
#pragma unroll
    for (int a = 0; a < 6; ++a) o.q[a] = S.ring[slot][a][t];
    o.e = e[slot];
  }
};

// ---------------------------------------------------------------------------
// block sums: one warp per value adds the values of the nw warps that have it (the block's
// first) and writes the block's partial.  An
// FP64 addition of a warp, whatever it adds, occupies the SM's FP64 pipe for 19 cycles.
// Blocks of up to 256 threads
// ---------------------------------------------------------------------------
template <int NV, int NT>
struct FxSumBuf {
  zd v[NV][NT];
};
template <int NV, int NT>
__device__ __forceinline__ void fx_block_partials(const zd (&v)[NV], FxSumBuf<NV, NT>& buf, zd* part, int nw) {
#pragma unroll
  for (int i = 0; i < NV; ++i) buf.v[i][threadIdx.x] = v[i];
  __syncthreads();
  const int lane = threadIdx.x & 31;
  for (int i = threadIdx.x >> 5; i < NV; i += blockDim.x >> 5) {
    const zd* q = &buf.v[i][lane];
    zd s = q[0];
    for (int t = 1; t < nw; ++t) s = s + q[32 * t];
    s = warp_sum(s);
    if (lane == 0) part[i * gridDim.x + blockIdx.x] = s;
  }
}

// The sums of the n blocks' partials (per value in block order per thread, then a fixed tree),
// in every lane of warp 0; every thread of the block calls it.  The order depends on n and on
// the number nw of warps that take part.  The values are spread over the
// warps, a value over several only where each has partials (trees and sums of nothing cost as
// much FP64 pipe as others), and eight loads per thread are in flight at a time.  Two values of
// 608 blocks took 8700 cycles with all warps at one value after the other; a call at 14x14^3,
// k = 800 402 -> 393 ms, at 4x4^3, k = 200 23.9 -> 22.7 ms.
template <int NV>
__device__ __forceinline__ void fx_sum_partials(const zd* part, int n, zd (&out)[NV], zd* scratch, int nw) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int per = max(1, min(nw / NV, (n + 31) >> 5));   // warps per value
  const int h = w % per;
  for (int i = w / per; i < NV && w < nw / per * per; i += nw / per) {
    const zd* p = part + (int64_t)i * n;
    zd v = mk(0.0, 0.0), v1 = mk(0.0, 0.0);   // two chains: an addition's latency is long
    for (int b0 = h * 32; b0 < n; b0 += 8 * 32 * per) {
      zd t[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int b = b0 + u * 32 * per + lane;
        t[u] = b < n ? ld_cg(p + b) : mk(0.0, 0.0);
      }
#pragma unroll
      for (int u = 0; u < 8; u += 2) {
        if (b0 + u * 32 * per < n) v = v + t[u];
        if (b0 + (u + 1) * 32 * per < n) v1 = v1 + t[u + 1];
      }
    }
    v = warp_sum(n > 32 * per ? v + v1 : v);
    if (lane == 0) scratch[i * 32 + h] = v;
  }
  __syncthreads();
  if (w == 0) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      out[i] = scratch[i * 32];
      for (int q = 1; q < per; ++q) out[i] = out[i] + scratch[i * 32 + q];
    }
  }
}

}  // namespace ov
