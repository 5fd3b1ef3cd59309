// wide.cuh — floating point with a 128-bit significand on the integer pipe,
// for the k-by-k steps of the compensated modes.
//
// These steps (Cholesky and Jacobi of the Gram matrix, arXiv:1806.01036, Sec.
// 4.2) need at least double-double accuracy.  On this GPU double-double itself
// is the slow way to it: the FP64 pipe does 2 FMA per clock and SM with a
// latency of 65 cycles, so a double-double addition is about 13 dependent FP64
// operations = 850 cycles, while 32-bit integer multiply-adds run at 64 lanes
// per clock with a latency of a few cycles.  A wide number is
//     (-1)^s m 2^(e - 127),  2^127 <= m < 2^128, or zero (m = 0).
// Operations truncate; their relative errors are below 2^-119 (products and
// sums of two products 2^-123 of the larger product), double-double's are
// about 2^-104.
// Exponents are plain integers: nothing over- or underflows before the
// conversion back to double-double.
#pragma once

#include "fx.cuh"

namespace eo {
namespace fx {

struct wide {
  u128 m;
  int e, s;
};

constexpr int kWideZero = -(1 << 28);  // exponent of zero (sums of two of them stay far below any other)

FX_HD wide wide_zero() { return wide{0, kWideZero, 0}; }
FX_HD wide wide_one() { return wide{(u128)1 << 127, 0, 0}; }
FX_HD wide wide_neg(wide a) { return wide{a.m, a.e, a.s ^ 1}; }
FX_HD bool wide_is_zero(wide a) { return (unsigned long long)(a.m >> 64) == 0ull; }

FX_HD unsigned long long mulhi64(unsigned long long a, unsigned long long b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (unsigned long long)(((u128)a * b) >> 64);
#endif
}

// High 128 bits of a 256-bit product, less at most 3 units (the low halves'
// product and two carries are left out).
FX_HD u128 mulhi128(u128 a, u128 b) {
  const unsigned long long a1 = (unsigned long long)(a >> 64), a0 = (unsigned long long)a;
  const unsigned long long b1 = (unsigned long long)(b >> 64), b0 = (unsigned long long)b;
  return (u128)a1 * b1 + mulhi64(a1, b0) + mulhi64(a0, b1);
}

// v >> n for n >= 0 (0 from 128 on).
FX_HD u128 shr128(u128 v, int n) {
  const unsigned long long h = (unsigned long long)(v >> 64), l = (unsigned long long)v;
  const int r = n & 63;
  const unsigned long long hs = h >> r, ls = (l >> r) | ((h << 1) << (63 - r));
  const unsigned long long h1 = n < 64 ? hs : 0ull, l1 = n < 64 ? ls : hs;
  return n < 128 ? ((u128)h1 << 64) | l1 : (u128)0;
}

// The number of magnitude u 2^(x - 127) (any u) and sign s.
FX_HD wide wide_norm(u128 u, int x, int s) {
  unsigned long long h = (unsigned long long)(u >> 64), l = (unsigned long long)u;
  if (h == 0ull) {  // cancelled by 64 bits or more: rare
    if (l == 0ull) return wide_zero();
    h = l;
    l = 0ull;
    x -= 64;
  }
  const int z = clz64(h);
  return wide{((u128)((h << z) | ((l >> 1) >> (63 - z))) << 64) | (l << z), x - z, s};
}

FX_HD wide wide_mul(wide a, wide b) {
  const u128 p = mulhi128(a.m, b.m);  // in [2^126 - 3, 2^128), or zero
  const int up = 1 - (int)(p >> 127);
  wide r{p << up, a.e + b.e + 1 - up, a.s ^ b.s};
  if ((unsigned long long)(p >> 64) == 0ull) r = wide_zero();
  return r;
}

// +-P 2^(ep - 127) +- Q 2^(eq - 127) with P, Q < 2^126
FX_HD wide wide_sum(u128 P, int ep, int sp, u128 Q, int eq, int sq) {
  const int d = ep - eq;
  P = shr128(P, d < 0 ? -d : 0);
  Q = shr128(Q, d > 0 ? d : 0);
  const i128 r = (i128)P + (sp != sq ? -(i128)Q : (i128)Q);
  const bool neg = r < 0;
  return wide_norm(neg ? (u128)(-r) : (u128)r, d < 0 ? eq : ep, sp ^ (int)neg);
}
FX_HD wide wide_add(wide a, wide b) { return wide_sum(a.m >> 2, a.e + 2, a.s, b.m >> 2, b.e + 2, b.s); }
FX_HD wide wide_sub(wide a, wide b) { return wide_add(a, wide_neg(b)); }
// a x + b y, aligned as products (the error is relative to the larger product)
FX_HD wide wide_dot2(wide a, wide x, wide b, wide y) {
  // a product's high half p has the value p 2^(ea + ex - 126): p >> 2 at exponent ea + ex + 3
  return wide_sum(mulhi128(a.m, x.m) >> 2, a.e + x.e + 3, a.s ^ x.s, mulhi128(b.m, y.m) >> 2, b.e + y.e + 3, b.s ^ y.s);
}
FX_HD wide wide_fma(wide a, wide b, wide c) { return wide_add(wide_mul(a, b), c); }

// Top bits of m as a float in [1, 2].
FX_HD float wide_top(wide a) { return (float)(unsigned)(a.m >> 96) * 0x1p-31f; }

FX_HD float seed_rsqrt(float x) {
#ifdef __CUDA_ARCH__
  return rsqrtf(x);
#else
  return 1.0f / sqrtf(x);
#endif
}

// g^(-1/2) 2^127 for g in [1, 4), G = g 2^126: a float seed (|error| < 2^-20),
// a cubic step in 64 bits, a quadratic step in 128.  With e = 1 - g y^2,
// g^(-1/2) = y (1 + e/2 + 3 e^2/8 + ...).
FX_HD u128 rsqrt_fixed(u128 G, float g) {
  const unsigned long long y0 = (unsigned long long)(unsigned)(seed_rsqrt(g) * 0x1p31f) << 32;  // units 2^-63
  const unsigned long long g64 = (unsigned long long)(G >> 64);                                 // units 2^-62
  const long long e0 = (1ll << 60) - (long long)mulhi64(g64, mulhi64(y0, y0));                  // units 2^-60
  const long long f0 = e0 >> 8;                                                                 // units 2^-52
  const long long c0 = (e0 >> 1) + (((f0 * f0) >> 44) * 3 >> 3);
  const unsigned long long y1 = y0 + (unsigned long long)(long long)(((i128)y0 * c0) >> 60);
  const i128 e1 = ((i128)1 << 124) - (i128)mulhi128(G, (u128)y1 * y1);  // units 2^-124, below 2^-57
  return ((u128)y1 << 64) + (u128)(((i128)y1 * (long long)(e1 >> 5)) >> 56);
}

// 1 / sqrt(a), a > 0
FX_HD wide wide_rsqrt(wide a) {
  const int odd = a.e & 1;
  const u128 y = rsqrt_fixed(odd ? a.m : a.m >> 1, wide_top(a) * (odd ? 2.0f : 1.0f));  // (1/2, 1] 2^127
  return wide_norm(y, -(a.e - odd) / 2, 0);
}
FX_HD wide wide_sqrt(wide a) { return wide_is_zero(a) ? wide_zero() : wide_mul(a, wide_rsqrt(a)); }

// 1 / a, a != 0: a float seed, a cubic step in 64 bits, a quadratic step in 128.
FX_HD wide wide_recip(wide a) {
  const unsigned long long m1 = (unsigned long long)(a.m >> 64), m0 = (unsigned long long)a.m;
  if (m1 == 1ull << 63 && m0 == 0ull) return wide{a.m, -a.e, a.s};  // a power of two
  const unsigned long long y0 = (unsigned long long)(unsigned)(1.0f / wide_top(a) * 0x1p31f) << 32;  // units 2^-63
  const long long e0 = (1ll << 62) - (long long)mulhi64(m1, y0);                                     // units 2^-62
  const long long f0 = e0 >> 10;                                                                     // units 2^-52
  const unsigned long long y1 = y0 + (unsigned long long)(long long)(((i128)y0 * (e0 + ((f0 * f0) >> 42))) >> 62);
  const i128 e1 = ((i128)1 << 126) - (i128)((u128)m1 * y1 + mulhi64(m0, y1));  // units 2^-126, below 2^-59
  const u128 y = ((u128)y1 << 64) + (u128)(((i128)y1 * (long long)(e1 >> 5)) >> 57);
  return wide_norm(y, -a.e, a.s);
}

// A finite double-double (|lo| <= ulp(hi) / 2) as a wide number.
FX_HD wide wide_from(double hi, double lo) {
  auto parts = [](double x, u128& m, int& e) {  // |x| = m 2^(e - 127), m 2^75-aligned 53 bits
    const unsigned h = hi32(x);
    const int be = (int)((h >> 20) & 0x7ffu);
    m = ((u128)((h & 0xfffffu) | (be ? 0x100000u : 0u)) << 107) | ((u128)lo32(x) << 75);
    e = (be ? be : 1) - 1023;
  };
  u128 mh, ml;
  int eh, el;
  parts(hi, mh, eh);
  parts(lo, ml, el);
  // (a zero high part has exponent -1022 and its low part is zero)
  return wide_sum(mh >> 2, eh + 2, (int)(hi32(hi) >> 31), ml >> 2, el + 2, (int)(hi32(lo) >> 31));
}
// hi = the nearest double, lo = the nearest to the rest.
FX_HD void wide_to_dd(wide a, double& hi, double& lo) {
  const i128 w = (i128)(a.m >> 1);
  w_to_dd(a.s ? -w : w, a.e - 126, hi, lo);
}

// a > b in magnitude
FX_HD bool wide_abs_gt(wide a, wide b) { return a.e != b.e ? a.e > b.e : a.m > b.m; }

}  // namespace fx
}  // namespace eo
