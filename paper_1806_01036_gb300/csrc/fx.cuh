// fx.cuh — exact fixed-point accumulation of FP64 products on the integer pipe.
//
// The compensated ("DD") mode of arXiv:1806.01036, Sec. 4.2 needs sums of
// FP64 products accurate to about 2^-104 relative.  GB300 runs FP64 at about
// 2 FMA/clk/SM, but 32x32->64-bit integer multiply-adds (IMAD.WIDE) at about
// 64/clk/SM, so the sums are formed here in integer arithmetic, exactly,
// instead of with FP64 error-free transformations:
//
//  * A group of doubles that is summed over (a column of a row panel, a row
//    of V, a column of Z) shares one alignment exponent A = the largest
//    biased exponent in the group.  Each member x becomes the integer
//      X = floor(|x| * 2^(1126 - A)) < 2^104   (x ~= sign(x) * X * 2^(A - 1126)),
//    which is exact for every member within 51 binades of the largest, and
//    is split into four signed 26-bit limbs L_0..L_3 (L_0 most significant).
//    (A is a biased exponent: |x| < 2^(A - 1022), so X < 2^104.)
//  * A product x*y is sum_{a,b} L_a(x) L_b(y) 2^(26(6-a-b)) * 2^(Ax+Ay-2252).
//    The ten limb products with a + b <= 3 are accumulated per diagonal
//    d = a + b into 64-bit integers (each product < 2^52: exact for up to
//    448 rows per accumulator); the dropped pairs contribute less than
//    6 * 2^-104 of max|x| * max|y| per product.
//  * Diagonal accumulators are combined into a 128-bit integer W in units of
//    2^(Ax+Ay-2148) and rounded to FP64, or to a double-double, with
//    round-to-nearest-even done in integer arithmetic.
//
// Integer sums are exact and associative, so every reduction built on this
// is independent of the order of its partial sums.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define FX_HD __host__ __device__ __forceinline__
#else
#define FX_HD inline
#endif

namespace eo {
namespace fx {

FX_HD unsigned hi32(double x) {
#ifdef __CUDA_ARCH__
  return (unsigned)__double2hiint(x);
#else
  unsigned long long b;
  memcpy(&b, &x, 8);
  return (unsigned)(b >> 32);
#endif
}
FX_HD unsigned lo32(double x) {
#ifdef __CUDA_ARCH__
  return (unsigned)__double2loint(x);
#else
  unsigned long long b;
  memcpy(&b, &x, 8);
  return (unsigned)b;
#endif
}
FX_HD double from_bits(unsigned long long b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double x;
  memcpy(&x, &b, 8);
  return x;
#endif
}
FX_HD int clz64(unsigned long long v) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)v);
#else
  return v ? __builtin_clzll(v) : 64;
#endif
}

constexpr int kLimbBits = 26;
constexpr long long kLimbMask = (1ll << kLimbBits) - 1;
constexpr int kRowsPerDrain = 384;  // rows a diagonal accumulator may absorb (< 448)
constexpr int kScaleOffset = 2148;  // value = W * 2^(Ax + Ay - 2148)

typedef __int128 i128;
typedef unsigned __int128 u128;

struct Limbs {
  int v[4];
};

// Biased exponent used for alignment: 1..2046 for finite nonzero values (1 for
// subnormals), 0 for zero, 2047 for Inf/NaN.
FX_HD int align_exp(double x) {
  const unsigned hi = hi32(x);
  const unsigned lo = lo32(x);
  const int be = (hi >> 20) & 0x7ff;
  if (be == 0) return ((hi & 0xfffffu) | lo) ? 1 : 0;
  return be;
}

// Limbs of floor(|x| 2^(1126 - A)) with the sign of x; requires A >= align_exp(x).
// X = m 2^t (t = 51 - (A - be) <= 51) is formed as a 128-bit integer and the
// limbs are cut from it with funnel shifts.
FX_HD Limbs to_limbs(double x, int A) {
  const unsigned hi = hi32(x);
  const unsigned lo = lo32(x);
  int be = (hi >> 20) & 0x7ff;
  unsigned mh = hi & 0xfffffu;
  if (be) mh |= 0x100000u; else be = 1;
  const unsigned long long m = ((unsigned long long)mh << 32) | lo;  // < 2^53
  const int t = 51 - (A - be);
  u128 X;
  if (t >= 0) X = (u128)m << t;
  else if (t > -64) X = (u128)(m >> (-t));
  else X = 0;
  const unsigned long long x0 = (unsigned long long)X, x1 = (unsigned long long)(X >> 64);
  Limbs L;
  L.v[3] = (int)(x0 & kLimbMask);
  L.v[2] = (int)((x0 >> 26) & kLimbMask);
  L.v[1] = (int)(((x0 >> 52) | (x1 << 12)) & kLimbMask);
  L.v[0] = (int)((x1 >> 14) & kLimbMask);
  if (hi >> 31) {
#pragma unroll
    for (int a = 0; a < 4; ++a) L.v[a] = -L.v[a];
  }
  return L;
}

// Limbs of a double-double h + l (|l| <= ulp(h)/2) aligned to A > align_exp(h):
// floor(|h + l| 2^(1126 - A)), computed exactly in 128-bit integers.
FX_HD Limbs to_limbs_dd(double h, double l, int A) {
  auto fixed = [A](double x) -> i128 {  // signed, truncated toward zero
    const unsigned hi = hi32(x);
    const unsigned lo = lo32(x);
    int be = (hi >> 20) & 0x7ff;
    unsigned mh = hi & 0xfffffu;
    if (be) mh |= 0x100000u; else be = 1;
    const unsigned long long m = ((unsigned long long)mh << 32) | lo;
    const int t = 51 - (A - be);
    u128 X;
    if (t >= 0) X = (u128)m << t;       // t <= 51 + (be_l - be_h) <= 51
    else if (t > -64) X = (u128)(m >> (-t));
    else X = 0;
    return (hi >> 31) ? -(i128)X : (i128)X;
  };
  i128 X = fixed(h) + fixed(l);
  const bool neg = X < 0;
  u128 U = neg ? (u128)(-X) : (u128)X;
  Limbs L;
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int p = 78 - kLimbBits * a;
    int v = (int)((U >> p) & (u128)kLimbMask);
    L.v[a] = neg ? -v : v;
  }
  return L;
}

// acc += a * b with a 32x32 -> 64-bit signed multiply-add (one IMAD.WIDE).
FX_HD void madw(long long& acc, int a, int b) {
#ifdef __CUDA_ARCH__
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
#else
  acc += (long long)a * b;
#endif
}

// acc[d] += sum_{a+b=d} x_a y_b for d = 0..3 (ten IMAD.WIDE).
FX_HD void mac(long long acc[4], const Limbs& x, const Limbs& y) {
  madw(acc[0], x.v[0], y.v[0]);
  madw(acc[1], x.v[0], y.v[1]);
  madw(acc[1], x.v[1], y.v[0]);
  madw(acc[2], x.v[0], y.v[2]);
  madw(acc[2], x.v[1], y.v[1]);
  madw(acc[2], x.v[2], y.v[0]);
  madw(acc[3], x.v[0], y.v[3]);
  madw(acc[3], x.v[1], y.v[2]);
  madw(acc[3], x.v[2], y.v[1]);
  madw(acc[3], x.v[3], y.v[0]);
}

// mac() on limbs held in int4 (x = L0, y = L1, z = L2, w = L3).
FX_HD void mac4(long long acc[4], const int4& x, const int4& y) {
  madw(acc[0], x.x, y.x);
  madw(acc[1], x.x, y.y);
  madw(acc[1], x.y, y.x);
  madw(acc[2], x.x, y.z);
  madw(acc[2], x.y, y.y);
  madw(acc[2], x.z, y.x);
  madw(acc[3], x.x, y.w);
  madw(acc[3], x.y, y.z);
  madw(acc[3], x.z, y.y);
  madw(acc[3], x.w, y.x);
}

// W in units of 2^(Ax+Ay-2148): acc0 2^52 + acc1 2^26 + acc2 + floor(acc3 2^-26).
FX_HD i128 acc_to_w(const long long acc[4]) {
  return ((i128)acc[0] << 52) + ((i128)acc[1] << 26) + (i128)acc[2] + (i128)(acc[3] >> 26);
}

// Divide the accumulated value by 2^sh (floor), as when the alignment
// exponent of one of its factors grows by sh.  The diagonals carry different
// weights, so the value is combined first and redistributed exactly:
// W' = floor(W 2^-sh) = acc0' 2^52 + acc2' with 0 <= acc2' < 2^52.
FX_HD void acc_shift(long long acc[4], int sh) {
  if (sh <= 0) return;
  i128 w = ((i128)acc[0] << 52) + ((i128)acc[1] << 26) + (i128)acc[2] + (i128)(acc[3] >> 26);
  w = sh >= 127 ? (w < 0 ? (i128)-1 : (i128)0) : (w >> sh);
  acc[0] = (long long)(w >> 52);
  acc[1] = 0;
  acc[2] = (long long)(w & (((i128)1 << 52) - 1));
  acc[3] = 0;
}

FX_HD i128 w_shift(i128 w, int sh) {
  if (sh <= 0) return w;
  return sh >= 127 ? (i128)0 : (w >> sh);
}

FX_HD int clz128(u128 u) {
  const unsigned long long h = (unsigned long long)(u >> 64);
  return h ? clz64(h) : 64 + clz64((unsigned long long)u);
}

// Bits dropped from the sums of `rows` products, each below 2^124 (1 + 2^-7), so
// that their total stays below 2^127: ceil(log2(rows)) - 2, none for four rows.
FX_HD int fold_bits(unsigned rows) {
  const int b = rows > 1u ? 64 - clz64(rows - 1u) : 0;
  return b > 2 ? b - 2 : 0;
}

// Double with magnitude m * 2^e2 (2^52 <= m < 2^53, or m == 0) and the given sign.
FX_HD double make_double(bool neg, unsigned long long m, int e2) {
  if (m == 0) return neg ? -0.0 : 0.0;
  const int be = e2 + 52 + 1023;
  if (be >= 1 && be <= 2046) {
    const unsigned long long bits =
        ((unsigned long long)neg << 63) | ((unsigned long long)be << 52) | (m & ((1ull << 52) - 1));
    return from_bits(bits);
  }
  if (be > 2046) return from_bits(((unsigned long long)neg << 63) | 0x7ff0000000000000ull);
  const double v = ldexp((double)m, e2);  // subnormal range: rare
  return neg ? -v : v;
}

// Round |u| * 2^S to 53 bits (nearest, ties to even).  Returns the rounded
// mantissa m (2^52 <= m < 2^53) and its exponent e2 (value = m * 2^e2), and the
// rounded value as an integer in units of 2^S when it fits (for remainders).
struct Rounded {
  unsigned long long m;
  int e2;
  u128 as_units;  // m * 2^(e2 - S), exact
  bool fits;
};

FX_HD Rounded round53(u128 u, int S) {
  Rounded r;
  const int p = 127 - clz128(u);
  if (p <= 52) {
    r.m = (unsigned long long)u << (52 - p);
    r.e2 = S + p - 52;
    r.as_units = u;
    r.fits = true;
    return r;
  }
  int sh = p - 52;
  unsigned long long m = (unsigned long long)(u >> sh);
  const u128 rem = u & (((u128)1 << sh) - 1);
  const u128 half = (u128)1 << (sh - 1);
  if (rem > half || (rem == half && (m & 1))) ++m;
  u128 units = (u128)m << sh;  // m may be 2^53 here; the shift keeps it exact
  r.fits = sh + 53 < 127;
  if (m >> 53) {
    m >>= 1;
    ++sh;
  }
  r.m = m;
  r.e2 = S + sh;
  r.as_units = units;
  return r;
}

// Nearest double to w * 2^S (ties to even).  The top 64 bits of |w| and a
// sticky bit for the rest decide the rounding; results outside the normal
// range take the general path.
FX_HD double w_to_double(i128 w, int S) {
  if (w == 0) return 0.0;
  const bool neg = w < 0;
  const u128 u = neg ? (u128)(-w) : (u128)w;
  const unsigned long long uh = (unsigned long long)(u >> 64), ul = (unsigned long long)u;
  int lz;
  unsigned long long t;
  bool sticky;
  if (uh) {
    lz = clz64(uh);
    t = lz ? (uh << lz) | (ul >> (64 - lz)) : uh;
    sticky = (ul << lz) != 0;
  } else {
    lz = 64 + clz64(ul);
    t = ul << (lz - 64);
    sticky = false;
  }
  // t holds bits p .. p - 63 of u, p = 127 - lz its top bit: m = bits p .. p - 52
  unsigned long long m = t >> 11;
  const unsigned long long rb = t & 0x7ffull;
  if (rb > 0x400ull || (rb == 0x400ull && (sticky || (m & 1ull)))) ++m;
  int e2 = S + (127 - lz) - 52;
  if (m >> 53) {
    m >>= 1;
    ++e2;
  }
  const int be = e2 + 52 + 1023;
  if (be < 1 || be > 2046) {
    const Rounded r = round53(u, S);
    return make_double(neg, r.m, r.e2);
  }
  return from_bits(((unsigned long long)neg << 63) | ((unsigned long long)be << 52) | (m & ((1ull << 52) - 1)));
}

// Nearest float to w * 2^S (ties to even), subnormals and overflow included: w
// rounded to odd in 53 bits, which a second rounding to 24 bits or fewer
// cannot tell from w itself.
FX_HD float w_to_float(i128 w, int S) {
  if (w == 0) return 0.0f;
  const u128 u = w < 0 ? (u128)(-w) : (u128)w;
  const int lz = clz128(u);
  const u128 v = u << lz;  // top bit at 127
  const unsigned long long t = (unsigned long long)(v >> 64);
  const unsigned long long m = (t >> 11) | (unsigned long long)((t & 0x7ffull) != 0ull || (unsigned long long)v != 0ull);
  const float f = (float)ldexp((double)m, S + 75 - lz);
  return w < 0 ? -f : f;
}

// Double-double (hi, lo) nearest to w * 2^S: hi = RN(w 2^S), lo = RN(w 2^S - hi).
FX_HD void w_to_dd(i128 w, int S, double& hi, double& lo) {
  if (w == 0) {
    hi = 0.0;
    lo = 0.0;
    return;
  }
  const bool neg = w < 0;
  const u128 u = neg ? (u128)(-w) : (u128)w;
  const Rounded r = round53(u, S);
  hi = make_double(neg, r.m, r.e2);
  const i128 rem = (i128)u - (i128)r.as_units;  // |rem| <= half an ulp of hi, exact
  lo = w_to_double(neg ? -rem : rem, S);
}

// y - w 2^S, rounded to nearest.
FX_HD double sub_round(double y, i128 w, int S) {
  if (w == 0) return y;
  const unsigned hi = hi32(y);
  const unsigned lo = lo32(y);
  int be = (hi >> 20) & 0x7ff;
  unsigned mh = hi & 0xfffffu;
  if (be) mh |= 0x100000u; else be = 1;
  const unsigned long long m = ((unsigned long long)mh << 32) | lo;
  if (m == 0) return -w_to_double(w, S);
  const int ey = be - 1075;  // y = +-m 2^ey
  int d = ey - S;
  int T = S;
  i128 ym;
  if (d > 72) {  // y dominates: coarsen the grid to 2^(ey - 72)
    const int sh = d - 72;
    w = w_shift(w, sh);
    T = S + sh;
    ym = (i128)m << 72;
  } else if (d >= 0) {
    ym = (i128)m << d;
  } else {
    // y has bits below the product's grid: move w onto y's grid when it fits,
    // otherwise (|w| too large to shift) drop y's bits below 2^S
    const u128 aw = w < 0 ? (u128)(-w) : (u128)w;
    if (clz128(aw) > 1 - d) {
      w <<= -d;
      T = S + d;
      ym = (i128)m;
    } else {
      ym = -d >= 64 ? (i128)0 : (i128)(m >> (-d));
    }
  }
  if (hi >> 31) ym = -ym;
  return w_to_double(ym - w, T);
}

// Branch-free forms of w_to_double and sub_round for the common case, so
// that a thread can interleave the roundings of several outputs: the same
// bits as those functions whenever ok is set; ok is cleared when the
// result is not a normal double, and (sub_round) when y is not a normal
// double or has bits below the grid 2^S, and the caller then takes the
// general function.
FX_HD double w_to_double_fast(i128 w, int S, bool& ok) {
  const bool neg = w < 0;
  const u128 u = neg ? (u128)(-w) : (u128)w;
  const unsigned long long uh = (unsigned long long)(u >> 64), ul = (unsigned long long)u;
  const int lz = uh ? clz64(uh) : 64 + clz64(ul);
  const u128 v = u << (lz & 127);  // top bit at 127 (u == 0: result replaced below)
  const unsigned long long t = (unsigned long long)(v >> 64);
  const bool sticky = (unsigned long long)v != 0ull;
  unsigned long long m = t >> 11;
  const unsigned long long rb = t & 0x7ffull;
  m += (unsigned long long)(rb > 0x400ull || (rb == 0x400ull && (sticky || (m & 1ull))));
  const int carry = (int)(m >> 53);
  m >>= carry;
  const int be = S + 1150 - lz + carry;  // e2 + 52 + 1023 with e2 = S + (127 - lz) - 52 + carry
  ok = u == 0 || (be >= 1 && be <= 2046);
  const unsigned long long bits =
      ((unsigned long long)neg << 63) | ((unsigned long long)(be & 0x7ff) << 52) | (m & ((1ull << 52) - 1));
  return u == 0 ? 0.0 : from_bits(bits);
}

FX_HD double sub_round_fast(double y, i128 w, int S, bool& ok) {
  const unsigned hi = hi32(y), lo = lo32(y);
  const int be = (int)((hi >> 20) & 0x7ffu);
  const unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
  const int d = be - 1075 - S;  // y = +-m 2^(S + d)
  // y dominating by more than 2^72: the product's grid coarsened to
  // 2^(S + d - 72), w truncated onto it (as sub_round does)
  const int sh = d > 72 ? d - 72 : 0;
  const i128 wc = sh >= 127 ? (i128)0 : (w >> sh);
  const u128 ym = (u128)m << (d < 0 ? 0 : (d > 72 ? 72 : d));
  const i128 r = ((hi >> 31) ? -(i128)ym : (i128)ym) - wc;
  bool okr;
  const double o = w_to_double_fast(r, S + sh, okr);
  ok = okr && be >= 1 && be <= 2046 && d >= 0;
  return o;
}

// ---- the same two roundings on 32-bit words, for results whose low bits are
// neither all zeros nor all ones (any but about 2^-25 of them, when the result
// is not exact).  Variable 128-bit shifts, the carry chain of a negation and
// the tie logic are most of the forms above; here words are selected and
// funnel-shifted, a negative value is complemented instead of negated and a
// truncation is left standing, both of which move the value by less than 64
// units of a 32-bit word below the rounding bits, and ok is cleared when that
// word is within 64 of wrapping (ties and exact results among them).
FX_HD unsigned funnel_l(unsigned lo, unsigned hi, int s) {  // high word of (hi:lo) << (s mod 32)
#ifdef __CUDA_ARCH__
  return __funnelshift_l(lo, hi, (unsigned)s);
#else
  s &= 31;
  return s ? (hi << s) | (lo >> (32 - s)) : hi;
#endif
}
FX_HD int clz32(unsigned v) {
#ifdef __CUDA_ARCH__
  return __clz((int)v);
#else
  return v ? __builtin_clz(v) : 32;
#endif
}
FX_HD unsigned word(u128 v, int i) { return (unsigned)(v >> (32 * i)); }
FX_HD u128 from_words(unsigned w3, unsigned w2, unsigned w1, unsigned w0) {
  return (u128)(((unsigned long long)w3 << 32) | w2) << 64 | (((unsigned long long)w1 << 32) | w0);
}

// (r + f) 2^S (0 <= f < 1, f = 0 if |r| < 2^92) with the sign flipped if flip
// has its top bit set.
FX_HD double w_to_double_lean(u128 r, int S, unsigned flip, bool& ok) {
  const unsigned neg = (unsigned)((int)word(r, 3) >> 31);
  const unsigned u3 = word(r, 3) ^ neg, u2 = word(r, 2) ^ neg, u1 = word(r, 1) ^ neg, u0 = word(r, 0) ^ neg;
  const bool top = u3 != 0u;
  const unsigned a = top ? u3 : u2, b = top ? u2 : u1, c = top ? u1 : u0, d = top ? u0 : neg;
  const int lz = clz32(a);
  const unsigned t2 = funnel_l(b, a, lz), t1 = funnel_l(c, b, lz), t0 = funnel_l(d, c, lz);
  const int be1 = S + (top ? 1149 : 1117) - lz;  // biased exponent - 1
  ok = a != 0u && (unsigned)be1 < 2045u && t0 + 64u >= 128u;
  const unsigned hi = (t2 >> 11) + ((unsigned)be1 << 20);
  const unsigned long long bits = (((unsigned long long)hi << 32) | funnel_l(t1, t2, 21)) + ((t1 >> 10) & 1u);
  return from_bits(bits ^ ((unsigned long long)((neg ^ flip) & 0x80000000u) << 32));
}

// r 2^S rounded to FP32, the same way.
FX_HD float w_to_float_lean(u128 r, int S, bool& ok) {
  const unsigned neg = (unsigned)((int)word(r, 3) >> 31);
  const unsigned u3 = word(r, 3) ^ neg, u2 = word(r, 2) ^ neg, u1 = word(r, 1) ^ neg, u0 = word(r, 0) ^ neg;
  const bool top = u3 != 0u;
  const unsigned a = top ? u3 : u2, b = top ? u2 : u1, c = top ? u1 : u0;
  const int lz = clz32(a);
  const unsigned t2 = funnel_l(b, a, lz), t1 = funnel_l(c, b, lz);
  const int be1 = S + (top ? 253 : 221) - lz;  // biased exponent - 1
  ok = a != 0u && (unsigned)be1 < 253u && t1 + 64u >= 128u;
  const unsigned bits = ((t2 >> 8) + ((t2 >> 7) & 1u) + ((unsigned)be1 << 23)) | (neg & 0x80000000u);
  float f;
#ifdef __CUDA_ARCH__
  f = __uint_as_float(bits);
#else
  memcpy(&f, &bits, 4);
#endif
  return f;
}

// x widened without the FP64 pipe (finite, zero and non-finite values alike).
FX_HD double widen(float x) {
  unsigned u;
#ifdef __CUDA_ARCH__
  u = __float_as_uint(x);
#else
  memcpy(&u, &x, 4);
#endif
  const unsigned m = u & 0x7fffffffu;
  if (m - 0x00800000u >= 0x7f000000u && m != 0u) return (double)x;  // subnormal, Inf, NaN
  const unsigned hi = (u & 0x80000000u) | (m ? (m >> 3) + (896u << 20) : 0u);
  return from_bits(((unsigned long long)hi << 32) | (m << 29));
}

// Does y dominate the grid 2^S by more than 2^72 of its units in its last place?
FX_HD bool dominates(double y, int S) { return (int)((hi32(y) >> 20) & 0x7ffu) - 1075 - S > 72; }

// y - w 2^S with w = raw - K; |w| < 2^122.  FAR: y may dominate the grid.
template <bool FAR>
FX_HD double sub_round_lean(double y, u128 raw, u128 K, int S, bool& ok) {
  const unsigned hi = hi32(y), lo = lo32(y);
  // sign(y) (y - w 2^S) = (|y| + g 2^S), g = -w for y >= 0 (the complement of
  // raw - K - 1), w for y < 0
  const unsigned pos = ~(unsigned)((int)hi >> 31);
  u128 g = raw - from_words(word(K, 3), word(K, 2), word(K, 1), word(K, 0) + (pos & 1u));
  unsigned g3 = word(g, 3) ^ pos, g2 = word(g, 2) ^ pos, g1 = word(g, 1) ^ pos, g0 = word(g, 0) ^ pos;
  const int be = (int)((hi >> 20) & 0x7ffu);
  const unsigned mh = (hi & 0xfffffu) | 0x100000u;
  int d = be - 1075 - S;  // |y| = m 2^(S + d)
  if (FAR) {  // y dominating: its last bit at 41 to 72 of a frame some words up
    const int k = d > 72 ? (d - 41) >> 5 : 0;
    const unsigned sx = (unsigned)((int)g3 >> 31);
    g0 = k == 0 ? g0 : k == 1 ? g1 : k == 2 ? g2 : k == 3 ? g3 : sx;
    g1 = k == 0 ? g1 : k == 1 ? g2 : k == 2 ? g3 : sx;
    g2 = k == 0 ? g2 : k == 1 ? g3 : sx;
    g3 = k == 0 ? g3 : sx;
    d -= 32 * k;
    S += 32 * k;
  }
  const unsigned m0 = lo << (d & 31), m1 = funnel_l(lo, mh, d), m2 = funnel_l(mh, 0u, d);
  const bool w0 = d < 32, w1 = d < 64;
  const u128 ym = from_words(w0 ? 0u : w1 ? m2 : m1, w0 ? m2 : w1 ? m1 : m0, w0 ? m1 : w1 ? m0 : 0u, w0 ? m0 : 0u);
  bool okr;
  const double o = w_to_double_lean(ym + from_words(g3, g2, g1, g0), S, hi, okr);
  ok = okr && (unsigned)(be - 1) < 2046u && (unsigned)d <= 72u;
  return o;
}

// 256-bit signed accumulator for sums of 128-bit terms.
struct Acc256 {
  u128 lo;
  i128 hi;
  FX_HD void zero() {
    lo = 0;
    hi = 0;
  }
  FX_HD void add(i128 v) {
    const u128 nl = lo + (u128)v;
    hi += (v < 0 ? (i128)-1 : (i128)0) + (nl < lo ? (i128)1 : (i128)0);
    lo = nl;
  }
  FX_HD void add(const Acc256& o) {
    const u128 nl = lo + o.lo;
    hi += o.hi + (nl < lo ? (i128)1 : (i128)0);
    lo = nl;
  }
  // Reduce to a 128-bit value and an extra scale shift (truncating if needed).
  FX_HD i128 narrow(int& extra) const {
    const i128 top = (i128)lo >> 127;  // sign extension of lo as signed
    if (hi == top && (((i128)lo < 0) == (hi < 0))) {
      extra = 0;
      return (i128)lo;
    }
    // find how many bits the 256-bit value needs and shift right to fit in 126
    const bool neg = hi < 0;
    u128 mh = (u128)hi, ml = lo;
    if (neg) {  // magnitude of the two's complement 256-bit value
      ml = ~ml + 1;
      mh = ~mh + (ml == 0 ? 1 : 0);
    }
    const int bits = 128 + (128 - clz128(mh));
    const int sh = bits - 126;
    const u128 mag = (ml >> sh) | (mh << (128 - sh));
    extra = sh;
    return neg ? -(i128)mag : (i128)mag;
  }
};

}  // namespace fx
}  // namespace eo
