// Integer fixed-point helpers for the complex128 sweep arithmetic.
//
// The state inside a call is int64 with value = integer * 2^-S; unit-modulus factors
// (phases, mixer diagonals) are Q62 (value = integer * 2^-62).  Every helper uses
// integer instructions only (GB300's float64 pipe retires ~1.75 FMA per SM clock).
// The header compiles for the device and, for the CPU tests, for the host.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define QAOA_HD __host__ __device__ __forceinline__
#else
#define QAOA_HD inline
#endif

namespace qaoa {
namespace fx {

typedef __int128 i128;

QAOA_HD int clz64(unsigned long long a) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)a);
#else
  return a ? __builtin_clzll(a) : 64;
#endif
}

QAOA_HD double bits_to_double(unsigned long long b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  union {
    unsigned long long u;
    double d;
  } c;
  c.u = b;
  return c.d;
#endif
}

QAOA_HD float bits_to_float(unsigned b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  union {
    unsigned u;
    float f;
  } c;
  c.u = b;
  return c.f;
#endif
}

QAOA_HD float fma_f32(float a, float b, float c) {
#ifdef __CUDA_ARCH__
  return __fmaf_rn(a, b, c);
#else
  return __builtin_fmaf(a, b, c);
#endif
}

// x << s, zero from s = 64 on
QAOA_HD unsigned long long shl64(unsigned long long x, unsigned s) {
#ifdef __CUDA_ARCH__
  unsigned long long r;
  asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
  return r;
#else
  return s < 64 ? x << s : 0;
#endif
}

QAOA_HD unsigned long long double_to_bits(double d) {
#ifdef __CUDA_ARCH__
  return (unsigned long long)__double_as_longlong(d);
#else
  union {
    unsigned long long u;
    double d;
  } c;
  c.d = d;
  return c.u;
#endif
}

// round(v / 2^s) for s >= 0, ties toward +infinity
QAOA_HD long long round_shift(i128 v, int s) {
  return s > 0 ? (long long)((v + ((i128)1 << (s - 1))) >> s) : (long long)v;
}

// A value split into 32-bit limbs x = h * 2^32 + l with l signed, |l| <= 2^31 (8-byte
// aligned, so a prepared factor in shared memory loads as three 64-bit words).
struct alignas(8) Limbs {
  int h;
  int l;
};

QAOA_HD Limbs split(long long x) {
  const unsigned int l = (unsigned int)(unsigned long long)x;
  Limbs r;
  r.l = (int)l;
  r.h = (int)((unsigned int)((unsigned long long)x >> 32) + (l >> 31));  // a negative l borrows one from h
  return r;
}

// a * b + c for 32-bit a, b and a 64-bit c.  On the device this is one multiply-add-wide
// instruction; written as (long long)a * b + c the compiler emits a 64 x 64-bit multiply
// (measured: 8 instead of 3 instructions per product, 74 instead of 42 per complex multiply).
QAOA_HD long long madw(int a, int b, long long c) {
#ifdef __CUDA_ARCH__
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
#else
  return (long long)a * b + c;
#endif
}

// round((a b + c d) / 2^(62 + e)) for a, c with |.| < 2^61 and b, d Q62 with |.| <= 2^62,
// 0 <= e <= 30, from eight 32x32 -> 64-bit products.  x y = xh yh 2^64 + (xh yl + xl yh) 2^32
// + xl yl; the low products enter only through their high words, so the result can differ
// from exact rounding by one unit when the exact value lies within 2^-29 units of a tie.
QAOA_HD long long dot2_q62(Limbs a, Limbs b, Limbs c, Limbs d, int e) {
  const long long P = madw(c.h, d.h, madw(a.h, b.h, 0));
  const long long M = madw(c.l, d.h, madw(c.h, d.l, madw(a.l, b.h, madw(a.h, b.l, 0))));
  const long long Lh = (madw(a.l, b.l, 0) >> 32) + (madw(c.l, d.l, 0) >> 32);
  const long long T = M + Lh;  // value = P 2^64 + T 2^32 (up to the dropped low words)
  if (e <= 2) return (long long)((unsigned long long)P << (2 - e)) + ((T + (1ll << (29 + e))) >> (30 + e));
  return (P + ((T + (1ll << (29 + e))) >> 32)) >> (e - 2);
}

// (a b + c d + half 2^32) / 2^64 rounded down, without the products of the low limbs: half
// starts the middle sum and the middle sum's high word starts the high sum, so rounding and
// carrying cost no additions of their own (a 64-bit add occupies the integer pipes as long as
// a product does; the complex multiplies of the sweeps lose 16 of their 32 add and shift
// instructions this way)
QAOA_HD long long dot2_hi64(Limbs a, Limbs b, Limbs c, Limbs d, long long half) {
  const long long T = madw(c.l, d.h, madw(c.h, d.l, madw(a.l, b.h, madw(a.h, b.l, half))));
  return madw(c.h, d.h, madw(a.h, b.h, T >> 32));
}

// dot2_q62 without the products of the low limbs: they add at most 2^(1 - e) result units,
// so for e >= 3 the result is within one unit of exact rounding (two fewer 32 x 32-bit
// products per call)
QAOA_HD long long dot2_q62_hi(Limbs a, Limbs b, Limbs c, Limbs d, int e) {
  if (e > 2) return dot2_hi64(a, b, c, d, 1ll << (29 + e)) >> (e - 2);
  const long long P = madw(c.h, d.h, madw(a.h, b.h, 0));
  const long long T = madw(c.l, d.h, madw(c.h, d.l, madw(a.l, b.h, madw(a.h, b.l, 1ll << (29 + e)))));
  return (long long)((unsigned long long)P << (2 - e)) + (T >> (30 + e));
}

// Exact 128-bit products from four 32 x 32-bit limb products each (fused multiply-add-wide
// on the device).  Operands |.| < 2^61: the high limbs are below 2^29 in magnitude, so the
// middle sums stay inside int64; the low-limb difference (two products of magnitude <= 2^62)
// does too.
// a b - c d
QAOA_HD i128 dot2_exact(long long a, long long b, long long c, long long d) {
  const Limbs A = split(a), B = split(b), C = split(c), D = split(d);
  const long long P = madw(-C.h, D.h, madw(A.h, B.h, 0));
  const long long M = madw(A.h, B.l, madw(A.l, B.h, 0)) - madw(C.h, D.l, madw(C.l, D.h, 0));
  const long long L = madw(A.l, B.l, 0) - madw(C.l, D.l, 0);
  return ((i128)P << 64) + ((i128)M << 32) + (i128)L;
}
// a c for a 64-bit a (|a| < 2^62) and a 32-bit c
QAOA_HD i128 mul_wide32(long long a, int c) {
  const Limbs A = split(a);
  return ((i128)madw(A.h, c, 0) << 32) + (i128)madw(A.l, c, 0);
}

// x * u / 2^(62 + e) for complex x (|re|, |im| < 2^61) and a Q62 unit complex u
struct C64 {
  long long x, y;
};

QAOA_HD C64 cmul_q62(long long xr, long long xi, long long ur, long long ui, int e) {
  const Limbs r = split(xr), i = split(xi), ni = split(-xi);
  const Limbs a = split(ur), b = split(ui);
  C64 o;
  o.x = dot2_q62(r, a, ni, b, e);  // xr ur - xi ui
  o.y = dot2_q62(r, b, i, a, e);   // xr ui + xi ur
  return o;
}

// cmul_q62 with dot2_q62_hi (for e >= 3: within one unit of exact rounding)
QAOA_HD C64 cmul_q62_hi(long long xr, long long xi, long long ur, long long ui, int e) {
  const Limbs r = split(xr), i = split(xi), ni = split(-xi);
  const Limbs a = split(ur), b = split(ui);
  C64 o;
  o.x = dot2_q62_hi(r, a, ni, b, e);
  o.y = dot2_q62_hi(r, b, i, a, e);
  return o;
}

// Reference with 128-bit products (one rounding per part); any |x| < 2^63.
QAOA_HD C64 cmul_q62_exact(long long xr, long long xi, long long ur, long long ui, int e) {
  const i128 re = (i128)xr * ur - (i128)xi * ui;
  const i128 im = (i128)xr * ui + (i128)xi * ur;
  C64 o;
  o.x = round_shift(re, 62 + e);
  o.y = round_shift(im, 62 + e);
  return o;
}

// A Q62 unit complex number u = ur + i ui prepared for repeated multiplies: the limbs of ur,
// ui and -ui (the negation done once here instead of once per product).
struct Factor {
  Limbs r, i, ni;
};

QAOA_HD Factor factor(long long ur, long long ui) {
  Factor f;
  f.r = split(ur);
  f.i = split(ui);
  f.ni = split(-ui);
  return f;
}

// x * u / 2^(62 + e) with u given as a Factor (conjugated when CONJ): the real part is
// xr ur + xi (-ui), the imaginary part xr ui + xi ur (for conj(u): xr ur + xi ui and
// xr (-ui) + xi ur).  FULL keeps every limb product (within one unit of exact rounding,
// like cmul_q62); otherwise the low x low products are dropped: within one unit for
// e >= 3 and within three units for e = 0.
template <bool FULL, bool CONJ>
QAOA_HD C64 cmul_factor(long long xr, long long xi, const Factor& f, int e) {
  const Limbs r = split(xr), i = split(xi);
  const Limbs& ui = CONJ ? f.ni : f.i;
  const Limbs& nui = CONJ ? f.i : f.ni;
  C64 o;
  if (FULL) {
    o.x = dot2_q62(r, f.r, i, nui, e);
    o.y = dot2_q62(r, ui, i, f.r, e);
  } else {
    o.x = dot2_q62_hi(r, f.r, i, nui, e);
    o.y = dot2_q62_hi(r, ui, i, f.r, e);
  }
  return o;
}

// cmul_factor<false, false> for e >= 3, on limbs the caller has split
QAOA_HD C64 cmul_big(Limbs r, Limbs i, const Factor& f, int e) {
  C64 o;
  o.x = dot2_hi64(r, f.r, i, f.ni, 1ll << (29 + e)) >> (e - 2);
  o.y = dot2_hi64(r, f.i, i, f.r, 1ll << (29 + e)) >> (e - 2);
  return o;
}

// x * u / 2^62 (conj(u) when CONJ) for |re x|, |im x| <= 2^60: the operand is scaled by 4 first,
// so the rounded sum is the high word pair itself (no shift after the products) and the
// dropped low x low products stay below half a unit: within one unit of exact rounding.
template <bool CONJ>
QAOA_HD C64 cmul_unit(long long xr, long long xi, const Factor& f) {
  const Limbs r = split((long long)((unsigned long long)xr << 2)), i = split((long long)((unsigned long long)xi << 2));
  const Limbs& ui = CONJ ? f.ni : f.i;
  const Limbs& nui = CONJ ? f.i : f.ni;
  C64 o;
  o.x = dot2_hi64(r, f.r, i, nui, 1ll << 31);
  o.y = dot2_hi64(r, ui, i, f.r, 1ll << 31);
  return o;
}

// x c / 2^62 for |x| < 2^59 and a Q62 c with |c| <= 2^62, by cmul_unit's rounding (within one unit)
QAOA_HD long long mul_unit(long long x, Limbs c) {
  const Limbs a = split((long long)((unsigned long long)x << 2));
  return madw(a.h, c.h, madw(a.l, c.h, madw(a.h, c.l, 1ll << 31)) >> 32);
}

// Low x low part of w.x v.y - w.y v.x: its high word (rounded down) and its low word.  Limbs lie in
// [-2^31, 2^31), so the difference of the two products fits 64 bits.
QAOA_HD long long low_diff(Limbs vx, Limbs vy, Limbs wx, Limbs wy) {
  return madw(wx.l, vy.l, 0) - madw(wy.l, vx.l, 0);
}

// Running sums of Im(conj(w) v) = w.x v.y - w.y v.x by limb weight, exact: value = P 2^64 + M 2^32 + L,
// one multiply-add-wide per limb product and few carries (an exact 128-bit product and sum per term
// took ~80 instructions per amplitude, this ~17).  Leaving the four lowest bits of w out of the low x
// low products saved two of them, but those bits are all of w where amplitudes are small: the n = 20
// gradient of costs of 1e-6 was off by 8e-9 instead of 1e-10.
// Sums of up to 8 terms with weights 0..3 fit int64 when the 2-norms of w and of v over the
// terms are at most 1.1 x 2^60: |h| norms are then at most 1.1 x 2^28 and each of M's two
// halves at most that x 2^31 sqrt(2 sum of squared weights <= 48) < 2^62.
struct ImSum {
  unsigned long long P = 0, M = 0, L = 0;
  QAOA_HD void add(Limbs vx, Limbs vy, Limbs wx, Limbs wy) {
    const int nwyh = -wy.h, nvxh = -vx.h;
    const long long d = low_diff(vx, vy, wx, wy);
    P = (unsigned long long)madw(nwyh, vx.h, madw(wx.h, vy.h, (long long)P));
    M = (unsigned long long)madw(wy.l, nvxh, madw(nwyh, vx.l, madw(wx.l, vy.h, madw(wx.h, vy.l, (long long)M))));
    M += (unsigned long long)(d >> 32);
    L += (unsigned)d;
  }
  // this += m s for a small m (modulo 2^64: intermediate sums may wrap)
  QAOA_HD void add_times(const ImSum& s, int m) {
    if (m == 0) return;
    P += s.P * (unsigned long long)(long long)m;
    M += s.M * (unsigned long long)(long long)m;
    L += s.L * (unsigned long long)(long long)m;
  }
  QAOA_HD i128 value() const {
    return ((i128)(long long)P << 64) + ((i128)(long long)M << 32) + (i128)(long long)L;
  }
};

// sum of c Im(conj(w) v) / 2^32 for integer c, |c| <= 2^28, and |components| < 2^59 (up to 8 terms), each
// term rounded to nearest (rounding down shifts the n = 28 gradient by 2e-12 of its size): the term
// is P 2^64 + Q 2^32, the low products' share in Q, and each word of P and Q is weighted by c with one
// multiply-add-wide.
struct WeightedImSum {
  long long ph = 0, pl = 0, qh = 0, ql = 0;
  QAOA_HD void add(long long vx_, long long vy_, long long wx_, long long wy_, int c) {
    const Limbs vx = split(vx_), vy = split(vy_), wx = split(wx_), wy = split(wy_);
    const int nwyh = -wy.h, nvxh = -vx.h;
    const long long d = low_diff(vx, vy, wx, wy), carry = (d >> 32) + (long long)((unsigned)d >> 31);
    const Limbs Q = split(madw(wy.l, nvxh, madw(nwyh, vx.l, madw(wx.l, vy.h, madw(wx.h, vy.l, carry)))));
    const Limbs P = split(madw(nwyh, vx.h, madw(wx.h, vy.h, 0)));
    ph = madw(P.h, c, ph);
    pl = madw(P.l, c, pl);
    qh = madw(Q.h, c, qh);
    ql = madw(Q.l, c, ql);
  }
  QAOA_HD i128 value() const { return ((i128)ph << 64) + ((i128)pl << 32) + ((i128)qh << 32) + (i128)ql; }
};

// float64 of x * 2^-s, correctly rounded (round to nearest, ties to even), assembled from
// the binary64 layout sign | 11-bit biased exponent | 52-bit fraction.  The result must be
// a normal number.
QAOA_HD double to_double(long long x, int s) {
  if (x == 0) return 0.0;
  const unsigned long long sgn = x < 0 ? (1ull << 63) : 0ull;
  const unsigned long long a = x < 0 ? (unsigned long long)(-x) : (unsigned long long)x;
  const int lz = clz64(a);
  const unsigned long long m = a << lz;  // leading one at bit 63
  unsigned long long keep = m >> 11;     // 53 significant bits
  const unsigned long long rem = m & 0x7FFull;
  keep += (rem > 0x400ull) || (rem == 0x400ull && (keep & 1ull));
  int ex = (63 - lz) - s;
  if (keep >> 53) {
    keep >>= 1;
    ++ex;
  }
  return bits_to_double(sgn | ((unsigned long long)(ex + 1023) << 52) | (keep & ((1ull << 52) - 1)));
}

// float64 of an int128 v * 2^-s (a sticky shift to 62 bits, then to_double)
QAOA_HD double i128_to_double(i128 v, int s) {
  const bool neg = v < 0;
  const unsigned __int128 a = neg ? (unsigned __int128)(-v) : (unsigned __int128)v;
  const unsigned long long hi = (unsigned long long)(a >> 64), lo = (unsigned long long)a;
  long long q;
  int sh = 0;
  if (hi == 0 && (lo >> 62) == 0) {
    q = (long long)lo;
  } else {
    const int nbits = hi ? 128 - clz64(hi) : 64 - clz64(lo);
    sh = nbits - 62;
    const unsigned __int128 mask = (((unsigned __int128)1) << sh) - 1;
    q = (long long)(a >> sh) | ((a & mask) != 0 ? 1 : 0);
  }
  return to_double(neg ? -q : q, s - sh);
}

// round(d * 2^s) as int64 (half away from zero) for |d| 2^s <= 2^62 (a cost vector's largest entry
// meets the bound with equality when it is a power of two)
QAOA_HD long long from_double(double d, int s) {
  const unsigned long long bits = double_to_bits(d);
  const int ex = (int)((bits >> 52) & 0x7FF);
  if (ex == 0) return 0;  // zero or subnormal: below every resolution used here
  const long long m = (long long)((bits & ((1ull << 52) - 1)) | (1ull << 52));
  const int sh = ex - 1075 + s;  // value * 2^s = m * 2^sh
  long long r;
  if (sh >= 0) r = m << (sh > 10 ? 10 : sh);  // clamp; callers stay in range
  else if (sh > -64) r = (m >> (-sh)) + ((m >> (-sh - 1)) & 1);
  else r = 0;
  return (bits >> 63) ? -r : r;
}

// (d mod 1) * 2^64 as an unsigned turn count
QAOA_HD unsigned long long frac_turns(double d) {
  const unsigned long long bits = double_to_bits(d);
  const int ex = (int)((bits >> 52) & 0x7FF);
  if (ex == 0) return 0ull;
  const unsigned long long m = (bits & ((1ull << 52) - 1)) | (1ull << 52);
  const int sh = ex - 1075 + 64;  // d * 2^64 = m * 2^sh
  unsigned long long t;
  if (sh >= 64) t = 0ull;
  else if (sh >= 0) t = m << sh;  // wraps mod 2^64
  else if (sh > -64) t = (m >> (-sh)) + ((m >> (-sh - 1)) & 1ull);
  else t = 0ull;
  return (bits >> 63) ? (0ull - t) : t;
}

// 2 (d - rint(d)) in float32 from integer bits, for finite d.  From 2^-12 on the fraction of the turn is
// the mantissa shifted: its upper 23 bits (a float32 by its bits: a conversion takes eight cycles) plus
// the signed 32 below them by one fused multiply-add, so the sum rounds once (half a unit in the last
// place, as a float64 difference and its conversion do; three quarters below 2^-21 of a turn).  At +-1/2
// the sign may differ.  A smaller d is its own fraction, converted by its bits (below 2^-126: zero).
// No branches: n = 29, p = 5 complex64 layers with U(0, 1) weights take 16.9 ms, 17.6 with the second
// form behind one (16.6 with the turn truncated to 2^-32, which left phases below 2^-25 of a turn with
// few bits).
QAOA_HD float two_turns_f32(double d) {
  const unsigned long long b = double_to_bits(d);
  const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b, ex = (hi >> 20) & 0x7FFu;
  const unsigned long long t0 = shl64((b & ((1ull << 52) - 1)) | (1ull << 52), ex - 1011u);
  const unsigned long long t = hi >> 31 ? 0ull - t0 : t0;
  const int l = (int)(unsigned)(t >> 9);
  const int h = (int)((unsigned)(t >> 32) + 256u) >> 9;
  const float x = bits_to_float(0x4B400000u + (unsigned)h);  // 1.5 x 2^23 + h
  const float big = fma_f32((float)l, 0x1.0p-54f, fma_f32(x, 0x1.0p-22f, -3.0f));
  const unsigned mag = ((hi << 3) | (lo >> 29)) + ((lo >> 28) & 1u) - (895u << 23);  // 2 |d|, rounded
  const unsigned small = (ex < 897u ? 0u : mag & 0x7FFFFFFFu) | (hi & 0x80000000u);
  return ex < 1011u ? bits_to_float(small) : big;
}

// exp(-2 pi i t / 2^64) in Q62: two 256-entry tables (tt[k] = exp(-2 pi i k / 2^8), tt[256 + k] =
// exp(-2 pi i k / 2^16)) take the turn's nearest multiple of 2^-16, and the residual angle rho
// (at most pi 2^-16 = 2^-14.35) enters as (1 - rho^2/2) - i (rho - rho^3/6), to 2^-57: rho is cut to 44
// bits for its powers, which is 2^-58.3 of rho^2/2, and that to 2^-58; the next term, rho^4/24, is
// 2^-62.  The tables are 8 KB, so a sweep holds them in shared memory beside its cost tile;
// three 1024-entry tables with a first-order residual (to 2^-55) took three reads from L2 and two
// 128-bit complex products per amplitude.
template <class E>
QAOA_HD C64 turn_phase(unsigned long long t, const E* tt) {
  const unsigned k = (unsigned)((t + (1ull << 47)) >> 48);                  // modulo 2^16
  const long long r = (long long)(t - ((unsigned long long)k << 48));       // [-2^47, 2^47)
  const E a = tt[(k >> 8) & 255], b = tt[256 + (k & 255)];
  const Limbs ax = split(a.x), ay = split(a.y), bx = split(b.x), by = split(b.y), nby = split(-b.y);
  const long long ex = dot2_q62_hi(ax, bx, ay, nby, 0), ey = dot2_q62_hi(ax, by, ay, bx, 0);
  const long long rho = mul_unit(2 * r, split(3622009729038561421ll));      // 2 pi r 2^-64: pi/4 in Q62
  const int x = (int)(rho >> 18);
  const int h4 = (int)(madw(x, x, 0) >> 31);                                // rho^2 / 2, 2^-58 units
  const long long s = rho - (madw(x, h4 / 3, 0) >> 40);                     // rho - rho^3 / 6
  const Limbs X = split(ex), Y = split(ey);
  C64 o;
  o.x = ex - (madw(X.h, h4, 0) >> 26) + mul_unit(s, Y);
  o.y = ey - (madw(Y.h, h4, 0) >> 26) - mul_unit(s, X);
  return o;
}

}  // namespace fx
}  // namespace qaoa
