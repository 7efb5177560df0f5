// Fixed-point arithmetic of the integer-sum binary64 substep: exact dot products
// of 61-bit integers, exact weighted sums wider than 64 bits, their conversion to
// binary64 with one rounding, and exp by Tang's table method in fixed point.
//
// Why integers: an FP64-pipe instruction holds an SM sub-partition's pipe for
// about 78 cycles per warp on GB300 (measured at 2070 MHz: DFMA, DMUL and DADD
// 75-80, int64 <-> binary64 conversions 68), a 32 x 32 + 64 multiply-add 2.2, a
// 64-bit addition 2.3, a funnel shift 2.2, a count of leading zeros 8.6.  An
// exact three-term dot product below costs about 27 integer-pipe cycles plus 38
// for its conversion, against 235 as three DFMAs on converted operands.
//
// Everything here is plain integer code that compiles for the host as well.
#pragma once

#include <cuda_runtime.h>

namespace ac {

#define AC_HD __host__ __device__ __forceinline__

typedef unsigned long long fx_u64;

AC_HD int fx_clz(unsigned v) {  // 32 for v = 0
#ifdef __CUDA_ARCH__
    return __clz((int)v);
#else
    return v ? __builtin_clz(v) : 32;
#endif
}

// High word of (hi:lo) << n, 0 <= n <= 32.
AC_HD unsigned fx_shl_hi(unsigned lo, unsigned hi, int n) {
#ifdef __CUDA_ARCH__
    return __funnelshift_lc(lo, hi, n);
#else
    return n >= 32 ? lo : (n ? (hi << n) | (lo >> (32 - n)) : hi);
#endif
}

AC_HD unsigned fx_mulhi32(unsigned a, unsigned b) { return (unsigned)(((fx_u64)a * b) >> 32); }

AC_HD double fx_bits_to_double(long long b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double(b);
#else
    union { long long i; double d; } u;
    u.i = b;
    return u.d;
#endif
}

AC_HD long long fx_double_to_bits(double d) {
#ifdef __CUDA_ARCH__
    return __double_as_longlong(d);
#else
    union { long long i; double d; } u;
    u.d = d;
    return u.i;
#endif
}

// ---- exact dot products ------------------------------------------------------
// An operand x, |x| <= 2^60.8, as x = hi 2^32 + 2 lo (+ its lowest bit, dropped):
// both halves are signed 32-bit (0 <= lo < 2^31), so every partial product is one
// signed multiply-add into a 64-bit sum.
struct FxSplit {
    int hi, lo;
};
AC_HD FxSplit fx_split(long long x) {
    FxSplit s;
    s.hi = (int)(x >> 32);
    s.lo = (int)((unsigned)x >> 1);
    return s;
}

// Sum of up to three products: hh 2^64 + cr 2^33 + ll 4.  With |x| <= 2^60.8:
// |cr| <= 3 * 2 * 2^28.8 * 2^31 < 2^62.4 and ll <= 3 * 2^62 < 2^64.
struct FxDot {
    long long hh, cr;
    fx_u64 ll;
};
AC_HD FxDot fx_mul(FxSplit a, FxSplit b) {
    FxDot d;
    d.hh = (long long)a.hi * b.hi;
    d.cr = (long long)a.hi * b.lo + (long long)b.hi * a.lo;
    d.ll = (fx_u64)(unsigned)a.lo * (unsigned)b.lo;
    return d;
}
AC_HD void fx_mac(FxDot &d, FxSplit a, FxSplit b) {
    d.hh += (long long)a.hi * b.hi;
    d.cr += (long long)a.hi * b.lo;
    d.cr += (long long)b.hi * a.lo;
    d.ll += (fx_u64)(unsigned)a.lo * (unsigned)b.lo;
}

// A 96-bit signed value top 2^32 + low.
struct Fx96 {
    long long top;
    unsigned low;
};
// The dot product in units of 2^32 (its bits below 2^33 truncated).
AC_HD Fx96 fx_merge(const FxDot &d) {
    const long long t = d.cr + (long long)(d.ll >> 31);
    Fx96 v;
    v.top = d.hh + (t >> 31);
    v.low = (unsigned)t << 1;
    return v;
}
AC_HD Fx96 fx_dot3(const FxSplit (&a)[3], const FxSplit (&b)[3]) {
    FxDot d = fx_mul(a[0], b[0]);
    fx_mac(d, a[1], b[1]);
    fx_mac(d, a[2], b[2]);
    return fx_merge(d);
}
// a b - c e
AC_HD Fx96 fx_det2(FxSplit a, FxSplit b, FxSplit c, FxSplit e) {
    const FxDot p = fx_mul(a, b), q = fx_mul(c, e);
    const long long t = p.cr - q.cr + (long long)(p.ll >> 31) - (long long)(q.ll >> 31);
    Fx96 v;
    v.top = p.hh - q.hh + (t >> 31);
    v.low = (unsigned)t << 1;
    return v;
}

// ---- exact sums wider than 64 bits -----------------------------------------------
// H 2^32 + L, accumulated as w x for non-negative integer weights w < 2^15 and
// |x| < 2^62: L sums w times the low words (unsigned), H w times the high words.
struct FxWide {
    long long H;
    fx_u64 L;
};
AC_HD void fx_wmac(FxWide &a, long long x, int w) {
    a.L += (fx_u64)(unsigned)w * (unsigned)x;
    a.H += (long long)w * (int)(x >> 32);
}
AC_HD Fx96 fx_wide96(const FxWide &a) {
    Fx96 v;
    v.top = a.H + (long long)(a.L >> 32);
    v.low = (unsigned)a.L;
    return v;
}
// v >> S as 64 bits (0 < S < 32; the value must fit).
template <int S>
AC_HD long long fx_shift96(const Fx96 &v) {
    return (long long)(((fx_u64)v.top << (32 - S)) | (v.low >> S));
}

// x (rh 2^-31 + rl 2^-62), 0 <= rh, rl < 2^31: within a few units.
AC_HD long long fx_mulfrac(long long x, int rh, int rl) {
    const FxSplit s = fx_split(x);
    const long long cr = (long long)s.hi * rl + (long long)s.lo * rh;
    return 2 * ((long long)s.hi * rh + (cr >> 31));
}

// r in (0, 1] as hi 2^-31 + lo 2^-62 (1 as 1 - 2^-62).
inline void fx_fraction(double r, int *hi, int *lo) {
    *hi = *lo = 0x7fffffff;
    if (r < 1.0) {
        const double t = r * 2147483648.0;
        *hi = (int)t;
        *lo = (int)((t - (double)*hi) * 2147483648.0);
    }
}

// The normal binary64 with bits b in units of 2^(E - 1078), E at least its biased
// exponent: magnitude below 2^56 (truncated).  A zero or subnormal b gives 0 for E > 62.
AC_HD long long fx_align(long long b, int E) {
    const int e = (int)((b >> 52) & 0x7ff);
    const fx_u64 m = ((fx_u64)b & 0xfffffffffffffull) | 0x10000000000000ull;
    const int d = E - e;
    const long long x = (long long)((m << 3) >> (d > 63 ? 63 : d)), s = b >> 63;
    return (x ^ s) - s;
}

// ---- conversion -------------------------------------------------------------------
// v 2^e as binary64, rounded to nearest from the top 64 significant bits (a
// negative value is first replaced by its one's complement: half a unit of the
// 96 bits).  eb = e + FX_EB.
constexpr int FX_EB = 1023 + 95 - 1;
AC_HD double fx_to_double(const Fx96 &v, int eb) {
    const int th = (int)(v.top >> 32);
    const unsigned s = (unsigned)(th >> 31);
    unsigned h = (unsigned)th ^ s, m = (unsigned)v.top ^ s, l = v.low ^ s;
    const bool up = h == 0;  // the top word is empty: one word further down
    h = up ? m : h;
    m = up ? l : m;
    l = up ? 0u : l;
    // the middle word too: rare, but not rare enough to call it zero (a Laplacian on a
    // fine grid is some 2^53 units, one in 2^20 of them below 2^32)
    const bool up2 = h == 0;
    h = up2 ? m : h;
    m = up2 ? 0u : m;
    const int c = fx_clz(h);
    const unsigned H = fx_shl_hi(m, h, c), M = fx_shl_hi(l, m, c);  // top bit of H set
    const int e = eb - c - (up ? 32 : 0) - (up2 ? 32 : 0);
    fx_u64 b = (((fx_u64)H << 32) | M) >> 11;
    b += (M >> 10) & 1u;
    b += (fx_u64)(((unsigned)e << 20) + (s & 0x80000000u)) << 32;
    return fx_bits_to_double((int)H < 0 ? (long long)b : 0ll);
}
// x 2^e for a 64-bit x; eb = e + FX_EB64.
constexpr int FX_EB64 = FX_EB - 32;
AC_HD double fx_to_double(long long x, int eb) {
    Fx96 v;
    v.top = x;
    v.low = 0u;
    return fx_to_double(v, eb);
}

// ---- exp in fixed point ----------------------------------------------------------
// trunc(x 2^55) for |x| < 64.
AC_HD long long fx_from_double55(double x) {
    const long long b = fx_double_to_bits(x);
    const int eb = (int)((b >> 52) & 0x7ff);
    const fx_u64 m = ((fx_u64)b & 0xfffffffffffffull) | 0x10000000000000ull;
    int r = 1028 - eb;  // |x| = (m << 8) 2^-(61 - 6 + ...): (m << 8) >> r in units of 2^-55
    r = r > 63 ? 63 : r;
    const long long a = (long long)((m << 8) >> r);
    return b < 0 ? -a : a;
}

// exp(X 2^-55) for |X| < 2^61, by Tang's table method (ACM TOMS 15(2), 1989):
// N = floor(256 x / ln 2) = 256 m + j, r = x - N ln2/256 in [0, ln2/256), exp(x) =
// 2^m 2^(j/256) exp(r) with exp(r) - 1 from its degree-5 Taylor polynomial
// (truncation below 2^-60).  tab[j] = 2^(62 + j/256), l70 = 2^70 ln2/256.  Result
// within 0.6 ulp of exp of the fixed-point argument.
AC_HD double fx_exp55(long long X, const fx_u64 *tab, fx_u64 l70) {
    // N from the high word less one unit, so that r never comes out negative (r may
    // exceed ln2/256 by 2^-14 of it: the result's top bit is then taken below)
    const int xh = (int)(X >> 32) - 1;
    const int N = (int)(((long long)xh * 1549082004) >> 45);  // floor(256 / ln 2 * 2^22)
    const unsigned np = (unsigned)(N + 32768);
    fx_u64 r70 = ((fx_u64)X << 15) + 32768ull * l70;  // modulo 2^64: the result fits
    r70 -= (fx_u64)np * (unsigned)l70 + ((fx_u64)(np * (unsigned)(l70 >> 32)) << 32);
    const unsigned r40 = (unsigned)(r70 >> 30);
    const unsigned a36 = 2863311531u + fx_mulhi32(r40, 2236962u);       // 1/24 + r/120
    const unsigned b34 = 2863311531u + (fx_mulhi32(r40, a36) >> 10);    // 1/6 + r (..)
    const unsigned rh = (unsigned)(r70 >> 32), rl = (unsigned)r70;
    const fx_u64 rr76 = (fx_u64)rh * rh + (((fx_u64)rh * rl) >> 31);    // r^2
    const unsigned rr49 = (unsigned)(rr76 >> 27);
    const fx_u64 cube = (fx_u64)rr49 * fx_mulhi32(r40, b34);            // r^3 (..), 2^91
    const fx_u64 p70 = r70 + (rr76 >> 7) + (cube >> 21);                // exp(r) - 1
    const fx_u64 T = tab[N & 255];
    const unsigned Th = (unsigned)(T >> 32), Tl = (unsigned)T;
    const unsigned ph = (unsigned)(p70 >> 32), pl = (unsigned)p70;
    const fx_u64 tp = (fx_u64)Th * ph + (((fx_u64)Th * pl + (fx_u64)Tl * ph) >> 32);  // 2^68
    fx_u64 R = T + (tp >> 6);  // 2^(j/256) exp(r), 2^62
    int m = (N >> 8) + 1022;
    const bool over = (long long)R < 0;
    R = over ? R >> 1 : R;
    m += over ? 1 : 0;
    return fx_bits_to_double((long long)((R >> 10) + ((R >> 9) & 1u) + ((fx_u64)(unsigned)m << 52)));
}

}  // namespace ac
