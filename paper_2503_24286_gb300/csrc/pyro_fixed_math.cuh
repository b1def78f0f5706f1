// 64-bit fixed-point base-2 logarithms and exponentials on the integer pipe.
//
// Measured on GB300 (cycles of an SM per warp instruction): DFMA 16, IMAD.WIDE 1,
// IMAD 0.5, 64-bit add 0.6.  One FP64 operation costs as much as 16 wide
// multiplications, so the kernels that are bound by the FP64 pipe keep everything
// that lives in the logarithm of a rate -- Arrhenius exponents, Gibbs polynomials,
// concentrations -- in fixed point and come back to FP64 for the sums of rates
// only.  The fixed-point exponents are also finer than FP64 ones: an exponent near
// 2^6 has a unit of 2^-46 in FP64 and 2^-50 here.
//
// Formats (value = integer / 2^f):
//   lg   int64, f = 50: a base-2 logarithm, |value| < 8192.  The lowest bit is the
//        sign of the number (1: negative), so adding logarithms multiplies signs;
//        terms that carry no sign have it cleared.  Zero is LG_ZERO:
//        a product with one zero and a factor up to 2^1190 is below the smallest
//        double, and one of three zeros and a factor from 2^-770 stays in range.
//   frac int64, f = 63: a factor in [0, 1 - 2^-14].
//   coef int64, f = 51: a coefficient, |value| < 4096.
// Methods: exponential by a table of 2^(j/1024) and the Taylor series of 2^f
// (P.T.P. Tang, ACM TOMS 15(2), 1989); logarithm by a table of 256 reciprocals rc
// of 11 bits, for which m rc - 1 is exact in 64 bits, and the series of log2(1+t)
// (P.T.P. Tang, ACM TOMS 16(4), 1990).  The code also compiles as host C++ (the
// tests compare it with long double arithmetic there).
#pragma once

#if !defined(__CUDACC__) && !defined(__CUDACC_RTC__)
#include <cstring>
#endif

namespace pfx {

typedef long long i64;
typedef unsigned long long u64;

#if defined(__CUDACC__) || defined(__CUDACC_RTC__)
#define PFX_FN __device__ __forceinline__
PFX_FN unsigned mulhi_u(unsigned a, unsigned b) { return __umulhi(a, b); }
PFX_FN int mulhi_s(int a, int b) { return __mulhi(a, b); }
PFX_FN int clz64(u64 v) { return __clzll((long long)v); }
PFX_FN u64 dbits(double x) { return (u64)__double_as_longlong(x); }
PFX_FN double bitsd(u64 b) { return __longlong_as_double((long long)b); }
#else
#define PFX_FN inline
inline unsigned mulhi_u(unsigned a, unsigned b) { return (unsigned)(((u64)a * b) >> 32); }
inline int mulhi_s(int a, int b) { return (int)(((i64)a * b) >> 32); }
inline int clz64(u64 v) { return v ? __builtin_clzll(v) : 64; }
inline u64 dbits(double x) { u64 b; memcpy(&b, &x, 8); return b; }
inline double bitsd(u64 b) { double x; memcpy(&x, &b, 8); return x; }
#endif

constexpr int EXP2_TAB = 1024;     // 2^(j/1024) in [1, 2), unsigned, f = 63
constexpr int LOG2_TAB = 256;      // log2 entries
constexpr int LG_F = 50;
constexpr i64 LG_ZERO = -(2400ll << LG_F);
struct alignas(16) Log2Entry { i64 L; unsigned rc, pad; };   // -log2(rc/2048) (f = 62), rc

// v = hi 2^32 + lo with both halves signed, so that products of halves need no
// sign corrections
struct Pair { int hi, lo; };
PFX_FN Pair split(i64 v) {
  Pair p;
  p.lo = (int)v;
  p.hi = (int)((unsigned)((u64)v >> 32) + ((unsigned)p.lo >> 31));
  return p;
}

// c x for a coef and a frac: add + c x, f = 50 (rounded; the product of the low
// halves, below 2^-50, is left out)
PFX_FN i64 mul_add(Pair c, Pair x, i64 add) {
  i64 mid = (i64)c.hi * x.lo + 0x80000000ll;
  mid += (i64)c.lo * x.hi;
  return (i64)c.hi * x.hi + (add + (mid >> 32));
}

// Horner step q t + c for q, c of f = 50 and a frac t
PFX_FN i64 horner(i64 q, Pair t, i64 c) {
  const Pair a = split(q);
  i64 mid = (i64)a.hi * t.lo + 0x40000000ll;
  mid += (i64)a.lo * t.hi;
  const i64 h = (i64)a.hi * t.hi + (mid >> 32);    // f = 49
  return c + h + h;
}

// x in (0, 1 - 2^-14], a normal double, as a frac (truncated)
PFX_FN i64 frac_of(double x) {
  const u64 b = dbits(x);
  const int s = 1022 - (int)(b >> 52);             // -1 - exponent
  const u64 m = ((b & 0xfffffffffffffull) | 0x10000000000000ull) << 10;
  return s > 62 ? 0ll : (i64)(m >> s);
}

// a double of |y| < 2 with f = 61 (truncated; undefined beyond)
PFX_FN i64 fix61(double y) {
  const u64 b = dbits(y);
  const int s = 1024 - ((int)(b >> 52) & 0x7ff);
  const u64 m = ((b & 0xfffffffffffffull) | 0x10000000000000ull) << 10;   // f = 62, to shift by 1 - exponent
  const i64 v = s > 62 ? 0ll : (i64)(m >> (s & 63));
  return (b >> 63) ? -v : v;
}

// double of v 2^e, rounded (half up in magnitude), for results within the normal range
PFX_FN double scaled(i64 v, int e) {
  const u64 a = v < 0 ? (u64)(-v) : (u64)v;
  const int z = clz64(a | 1ull);
  const u64 m = a << z;                            // leading one at bit 63
  const u64 b = ((u64)(unsigned)(e + 63 - z + 1022) << 52) + (m >> 11) + ((m >> 10) & 1ull);
  return bitsd(a == 0 ? 0ull : (b | ((u64)v & 0x8000000000000000ull)));
}

// double of a value with f = 50 (truncated to 53 significant bits)
PFX_FN double to_double(i64 v) {
  const u64 a = v < 0 ? (u64)(-v) : (u64)v;
  const int z = clz64(a | 1ull);
  const u64 m = a << z;                            // leading one at bit 63
  const u64 e = (u64)(1023 + 63 - LG_F - z);
  const u64 b = (e << 52) + ((m << 1) >> 12);
  return bitsd(a == 0 ? 0ull : (b | ((u64)v & 0x8000000000000000ull)));
}

// Mantissa of 2^x for the fraction of a logarithm: 2^(x - floor x) as unsigned f = 63.
// Relative error below 2^-53.
PFX_FN u64 exp2_mant(i64 x, const u64* tab) {
  const u64 F = (u64)x << 24;                      // phi = F/2^64, f = phi/1024
  const unsigned Fh = (unsigned)(F >> 32), Fl = (unsigned)F;
  const u64 T = tab[(unsigned)((u64)x >> 40) & (EXP2_TAB - 1)];
  // 2^f - 1 = phi (C1 + phi (C2 + phi (C3 + phi C4)))/1024, C_i = ln2^i/i!/1024^(i-1)
  unsigned h = mulhi_u(Fh, 158u) + 931204u;                      // C4, C3: unit 2^-44
  h = mulhi_u(Fh, h) + 4127059964u;                              // C2
  const u64 G = (((u64)Fh * h) >> 12) + 0xb17217f7d1cf79acull;   // C1 + ..., f = 64
  const unsigned Gh = (unsigned)(G >> 32), Gl = (unsigned)G;
  const u64 P = (u64)Fh * Gh + ((u64)mulhi_u(Fh, Gl) + mulhi_u(Fl, Gh));
  const unsigned Th = (unsigned)(T >> 32), Tl = (unsigned)T, Ph = (unsigned)(P >> 32), Pl = (unsigned)P;
  const u64 Q = (u64)Th * Ph + ((u64)mulhi_u(Th, Pl) + mulhi_u(Tl, Ph));
  return T + (Q >> 10);
}

// 2^x with the sign in the lowest bit of x; 0 below 2^-1022, infinite from 2^1024
PFX_FN double exp2_lg(i64 x, const u64* tab) {
  const u64 m = exp2_mant(x, tab);
  const int n = (int)(x >> LG_F) + 1022;
  u64 b = ((m + 0x400ull) >> 11) + ((u64)(unsigned)n << 52);
  b = n < 0 ? 0ull : b;
  b = n > 2045 ? 0x7ff0000000000000ull : b;
  return bitsd(b | ((u64)x << 63));
}

// log2 of a mantissa m in [2^52, 2^53) read as m/2^52: f = 62, error below 2^-53
PFX_FN i64 log2_mant(u64 m, const Log2Entry* tab) {
  const Log2Entry E = tab[(unsigned)(m >> 44) & (LOG2_TAB - 1)];
  const i64 t = (i64)(m * E.rc - 0x8000000000000000ull);         // m rc/2^63 - 1, f = 63, |t| < 2^-8
  const i64 w = (i64)((u64)t << 8);                              // f = 64: w = 128 t
  const int wh = (int)(w >> 32);
  const unsigned wl = (unsigned)w;
  // log2(1+t) = (w/128) (d0 + w (d1 + w (d2 + w (d3 + w (d4 + w d5))))),
  // d_i = (-1)^i/(ln2 (i+1) 128^i)
  int f = mulhi_s(wh, -492) + 75639;                             // d5, d4: unit 2^-46
  f = mulhi_s(wh, f) - 12102203;                                 // d3
  f = mulhi_s(wh, f) + 2065442673;                               // d2
  const i64 e1 = (((i64)wh * f) >> 16) - 25989283394227192ll;    // d1 + ..., f = 62
  const int eh = (int)(e1 >> 32);
  const unsigned el = (unsigned)e1;
  // w e1 (f = 62): w is exact in 64 bits, its low half unsigned
  const i64 d = (i64)wh * eh + ((((i64)wh * (i64)(el >> 1)) >> 31) + (((i64)(wl >> 1) * eh) >> 31)) +
                6653256548922161246ll;                           // d0 + ..., f = 62
  const int dh = (int)(d >> 32);
  const unsigned dl = (unsigned)d;
  const i64 r = (i64)wh * dh + ((((i64)wh * (i64)(dl >> 1)) >> 31) + (((i64)(wl >> 1) * dh) >> 31));   // w d, f = 62
  return E.L + (r >> 7);
}

// lg of |x| for a normal double x > 0 (lowest bit clear)
PFX_FN i64 log2_of(double x, const Log2Entry* tab) {
  const u64 b = dbits(x);
  const int e = (int)(b >> 52) - 1023;
  const i64 l = log2_mant((b & 0xfffffffffffffull) | 0x10000000000000ull, tab);
  return ((i64)e << LG_F) + (((l + 0x1000ll) >> 13) << 1);
}

}  // namespace pfx
