// umma_rowprod.cu — compensated row products on the tcgen05 tensor cores:
//   projection  Y~ = Y - V C   (arXiv:1806.01036, Sec. 4.2, phase I, with
//                               C = V^T Y a double-double kv-by-k matrix);
//   update      Q  = X Z       (the final multiplication of phase II; Z the
//                               double-double R^{-1} or M^{-1/2}).
// Every output is the exact sum of its products (up to the dropped digit
// pairs), rounded once; the projection subtracts the exact sum from y before
// rounding.
//
// Digits (umma.cuh): a row of the streamed matrix (V or X) is aligned to its
// own largest exponent A_r, a column j of the small matrix (C or Z) to
// B_j = its largest exponent + 1 (room for the low part); both are cut into
// fourteen balanced 8-bit digits, of which the last four are zero for a row
// whose values lie within 25 binades ("near", nearly always).  A tile is 128
// rows = the 128 TMEM lanes; the K dimension is the kin columns of the row
// (kin <= 64), the N dimension the digit slab t and the output column j (16
// columns, padded).  One MMA multiplies digit slab s of the tile (M = 128, K =
// 16) by the slabs t = 0 .. 13 - s of the small matrix (N = 16 (14 - s)) and
// writes at TMEM column offset 16 s: column block d of a lane collects the
// digit diagonal d = s + t of its row.  A diagonal sum has at most kin x 14
// products of magnitude <= 2^14, below 2^24 for kin <= 64, so the FP32
// accumulators are exact over the whole row: a tile needs no drains, only an
// epilogue that combines its 14 diagonals per output in 32-bit words,
//   h = sum_d S_d 2^(8 (13 - d)),   sum_i v_i c_ij ~= h 2^(A_r + B_j - 2160),
// and rounds y - h 2^(...) (or h 2^(...)) to FP64 in integer arithmetic.  The
// dropped pairs (d >= 14: thirteen of weight 2^96 units^2 and fewer of smaller
// weights, max|v| >= 2^109 units, max|c| >= 2^108) are below 2^-103 max|v_i|
// max|c_ij| per product.
//
// Pipeline (one CTA per SM, tiles round-robin): the 16 converter warps hold a
// tile's values in registers (8 rows x 4 column groups per warp, coalesced
// along rows), fetched a tile ahead (staged through shared memory with cp.async
// for kin <= 32, loaded into registers after the previous tile's digits are
// stored for kin <= 64), find each row's exponent by shuffles, agree at the
// barrier that ends the previous tile whether every value of the tile is near,
// and write the digits in two groups of five slabs (a third of four for a tile
// that is not near) into two alternating shared-memory buffers; one warp issues
// the group's MMAs and commits them to an mbarrier per buffer; TMEM holds two
// accumulators, so the epilogue of tile i - 1 (tcgen05.ld, exact rounding,
// stores) runs while the tensor cores work on tile i (with two blocks of 16
// output columns, one accumulator each: see the kernel).  The projection's Y of
// a tile is prefetched into L2 a tile ahead and loaded before its epilogue
// reads TMEM.  Every wait is bounded (the outputs of a CTA whose wait ran out
// are NaN).  Each tile's loads precede its own stores, and no tile is written
// by another CTA, so the update may run in place.
//
// Bound by the integer pipe (57% busy over a kernel, saturated inside the
// conversion and the epilogue): 131 instructions an output and 40 to 60 a
// value; memory needs a third of the time.  Y - V C of 4e6 rows, with 7-bit
// digits and 128-bit roundings (280 instructions an output), then with 8-bit
// digits in byte places (ten near slabs and 14 diagonals, not twelve and 15),
// then with the diagonals combined in words and the lean roundings of fx.cuh,
// the outputs dealt evenly to the warps:
//   64 x 16 1.645 -> 1.507 -> 1.269 ms, 32 x 32 2.135 -> 1.933 -> 1.396,
//   32 x 16 1.230 -> 1.090 -> 0.829, 16 x 16 1.017 -> 0.907 -> 0.651,
//   20 x 4 0.969 -> 0.811 -> 0.601, 8 x 8 0.774 -> 0.687 -> 0.500.
// A launch's fixed part is about 8 us (64 x 16 on 1e4 rows: 14.4).
// Tiles that need all digits are no rare case for updates: a block whose columns
// span more than 25 binades has nothing else.  One CholQR pass on 4e6 rows, columns
// of one scale / over 10 decades, 7-bit digits first: 8 columns 1.19 / 1.19 -> 0.65 /
// 0.83 ms, 16 1.44 / 1.44 -> 0.94 / 1.12, 32 4.01 / 4.08 -> 2.51 / 3.10; Y - V C
// with 64 such columns of V 1.645 / 1.88 -> 1.269 / 1.96 (group 2 after the previous
// tile's epilogue; before it 1.22 / 2.11, with the third group's words formed anew
// 1.15 / 2.42: the more the rare path holds, the more the common one spills).
//
// FP32 updates (kin <= 32) take the same path with seven near slabs (24 bits
// and the near window); their outputs are rounded from the exact sum to FP32.
// 2e6 x 32: 4.0 ms on the FP64 pipe -> 0.57 ms.  Rows with a non-finite value, or
// with one that the 110 bits of the row's grid do not hold, are summed in FP64
// (plain_rows), so an Inf or NaN reaches the outputs whose sums it is part of
// (every row like that: 2e6 x 32 3.6 ms a call, all on the FP64 pipe 4.1), and
// all rows are when the columns' norms differ by more than 2^40 (kUneven).
#include <cuda_fp16.h>

#include <algorithm>
#include <cstdlib>
#include <type_traits>

#include "common.cuh"
#include "fx.cuh"
#include "umma.cuh"

namespace eo {
namespace {

using namespace fx;
using namespace umma;

constexpr int kConvWarps = 16;
constexpr int kConvThreads = 32 * kConvWarps;
constexpr int kThreads = kConvThreads + 32;  // plus one MMA-issuing warp
constexpr int kRows = 128;                   // rows per tile (MMA M, TMEM lanes)
constexpr int kOut = 16;                     // output columns of the MMA (padded)
constexpr int kGroup = 5;                    // digit slabs per group
constexpr int kGroupsNear = 2, kGroupsAll = 3;
// Slabs of a near tile: FP32 values have 24 bits, with the near window 49 of the 110.
template <typename Real>
constexpr int kNearOf = std::is_same_v<Real, float> ? 7 : kNear;
constexpr int kScaleProd = 2160;             // value of h: h 2^(A_r + B_j - 2160)
constexpr unsigned kAccCols = 256;           // TMEM columns per accumulator (224 used)
constexpr size_t kMinSmem = 120 * 1024;      // keeps one CTA per SM (TMEM: 512 columns)

// With kin <= 32 the digit buffers leave room below the shared-memory floor
// that keeps one CTA per SM: every converter thread then stages its own
// values of the next tile there (one buffer: a tile's values are read before
// the next tile's copies are issued into the same slots) while the current
// tile runs.  kin <= 64 has no room left (and smaller digit groups, to make
// some, cost more than the staging saves): there the next tile's values are
// loaded into registers once this tile's digits are stored (its values and
// digit words are dead then), so the loads are in flight during the
// previous tile's epilogue.
template <int W>
constexpr bool kStageValues = W <= 8;

// An accumulator S of magnitude below 2^22 becomes an integer with one FP32
// add: the bit pattern of 1.5 2^23 + S is 0x4B400000 + S, and two of them
// combine modulo 2^32 to S_2m 256 + S_2m+1 + kPairOffset, which stays in
// [0, 2^32) below 2^22.  A diagonal of kin <= 16 columns sums at most 14 x 16
// products of magnitude <= 2^14, below 2^22; wider rows pass 2^22 hardly ever,
// and the sum of the squares of the diagonals tells when one could.
constexpr unsigned kPairOffset = 0x8B400000u;
template <int W>
constexpr bool kSmallDiag = 4 * W * kAll * 16384 < 4194304;
constexpr float kSquares = 0x1p42f;  // the rounded sum of 14 squares; each |S| < 2^21.1
// The pairs' offsets in h: kPairOffset 2^(16 m), m = 0..6, modulo 2^128.
constexpr u128 offset_sum() {
  u128 k = 0;
  for (int m = 0; m < 7; ++m) k += (u128)kPairOffset << (16 * m);
  return k;
}
constexpr u128 kOffset = offset_sum();

__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

__device__ __forceinline__ void st_shared_v4(unsigned addr, unsigned a, unsigned b, unsigned c, unsigned d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void st_shared_v2(unsigned addr, unsigned a, unsigned b) {
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}

// h + kOffset from its pairs: the even pairs are its words, the odd ones lie half a word up.
__device__ __forceinline__ u128 pairs_sum(const unsigned (&q)[7]) {
  return from_words(q[0], q[2], q[4], q[6]) +
         from_words(q[1] >> 16, funnel_l(q[3], q[1], 16), funnel_l(q[5], q[3], 16), q[5] << 16);
}

// N groups of four TMEM columns (this warp's 32 lanes), 16 columns apart from column a on.
template <int N>
__device__ __forceinline__ void tmem_ld4(unsigned a, unsigned (&v)[N][4]) {
#pragma unroll
  for (int i = 0; i < N; ++i)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v[i][0]), "=r"(v[i][1]), "=r"(v[i][2]), "=r"(v[i][3])
                 : "r"(a + (unsigned)(i * kOut))
                 : "memory");
}
// Completes the loads into v (named, so that no use can move above the wait).
template <int N>
__device__ __forceinline__ void tmem_wait4(unsigned (&v)[N][4]) {
  static_assert(N == 2 || N == 4, "groups per load");
  if constexpr (N == 4)
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0][0]), "+r"(v[0][1]), "+r"(v[0][2]), "+r"(v[0][3]), "+r"(v[1][0]), "+r"(v[1][1]), "+r"(v[1][2]),
                   "+r"(v[1][3]), "+r"(v[2][0]), "+r"(v[2][1]), "+r"(v[2][2]), "+r"(v[2][3]), "+r"(v[3][0]), "+r"(v[3][1]),
                   "+r"(v[3][2]), "+r"(v[3][3])
                 :
                 : "memory");
  else
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0][0]), "+r"(v[0][1]), "+r"(v[0][2]), "+r"(v[0][3]), "+r"(v[1][0]), "+r"(v[1][1]), "+r"(v[1][2]),
                   "+r"(v[1][3])
                 :
                 : "memory");
}
// h + kOffset of four outputs from the columns tb, tb + 16, .., out of line: for
// diagonals that reach 2^22 (rare), and for outputs that the lean roundings left.
__device__ __noinline__ void combine_any(unsigned tb, u128* h) {
  unsigned q[4][7];
  float most = 0.f;
#pragma unroll
  for (int m = 0; m < 7; ++m) {
    unsigned v[2][4];
    tmem_ld4(tb + (unsigned)(2 * m * kOut), v);
    tmem_wait4(v);
#pragma unroll
    for (int y = 0; y < 4; ++y) {
      const float a = __uint_as_float(v[0][y]), b = __uint_as_float(v[1][y]);
      q[y][m] = __float_as_uint(a + 0x1.8p23f) * 256u + __float_as_uint(b + 0x1.8p23f);
      most = fmaxf(most, fmaxf(fabsf(a), fabsf(b)));
    }
  }
  if (!__any_sync(0xffffffffu, most >= 0x1p21f)) {
#pragma unroll
    for (int y = 0; y < 4; ++y) h[y] = pairs_sum(q[y]);
    return;
  }
  for (int y = 0; y < 4; ++y) h[y] = kOffset;
#pragma unroll 1
  for (int m = 0; m < 7; ++m) {
    unsigned v[2][4];
    tmem_ld4(tb + (unsigned)(2 * m * kOut), v);
    tmem_wait4(v);
    for (int y = 0; y < 4; ++y) {
      const long long r =
          (long long)__float2int_rn(__uint_as_float(v[0][y])) * 256 + __float2int_rn(__uint_as_float(v[1][y]));
      h[y] += (u128)(i128)r << (16 * (6 - m));
    }
  }
}

// The words of one slab for W values of a row, stored at dst (W = 16: two
// 16-byte chunks 128 bytes apart; W = 8: one chunk; W = 4: half a chunk).
template <int W>
__device__ __forceinline__ void st_slab(unsigned dst, const unsigned (&w)[W / 2]) {
  if constexpr (W == 16) {
    st_shared_v4(dst, w[0], w[1], w[2], w[3]);
    st_shared_v4(dst + 128u, w[4], w[5], w[6], w[7]);
  } else if constexpr (W == 8) {
    st_shared_v4(dst, w[0], w[1], w[2], w[3]);
  } else {
    st_shared_v2(dst, w[0], w[1]);
  }
}

// Lane words of W near values: z[m][i] holds digits 2i (high bytes) and 2i + 1
// (low bytes) of the pair m.
template <int W, bool ZERO>
__device__ __forceinline__ void near_lanes(const double (&v)[W], int A, unsigned (&z)[W / 2][5], unsigned (&sg)[W / 2]) {
#pragma unroll
  for (int m = 0; m < W / 2; ++m) {
    unsigned a1, a2, a3, b1, b2, b3;
    near_words<ZERO>(v[2 * m], 25 - A, a1, a2, a3);
    near_words<ZERO>(v[2 * m + 1], 25 - A, b1, b2, b3);
    sg[m] = sign2(v[2 * m], v[2 * m + 1]).mul;
    z[m][0] = __byte_perm(a3, b3, 0x5410);
    z[m][1] = __byte_perm(a2, b2, 0x7632);
    z[m][2] = __byte_perm(a2, b2, 0x5410);
    z[m][3] = __byte_perm(a1, b1, 0x7632);
    z[m][4] = __byte_perm(a1, b1, 0x5410);
  }
}
// Group G of near values: N slabs from 5 G on.
template <int G, int N, int W>
__device__ __forceinline__ void store_near(unsigned dst, unsigned slab_bytes, const unsigned (&z)[W / 2][5],
                                           const unsigned (&sg)[W / 2], unsigned e1024) {
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const int s = G * kGroup + j;
    unsigned w[W / 2];
#pragma unroll
    for (int m = 0; m < W / 2; ++m) {
      const Sign2 f{sg[m], hmul2(sg[m], s == 0 ? 0xE400E400u : 0xE480E480u)};
      w[m] = s % 2 == 0 ? digit_hi(z[m][s / 2], e1024, f) : digit_lo(z[m][s / 2], e1024, f);
    }
    st_slab<W>(dst + (unsigned)j * slab_bytes, w);
  }
}
// Lane words of any two values: y[i] holds digits 2i (high bytes) and 2i + 1 (low bytes).
__device__ __forceinline__ void any_lanes(double va, double vb, int A, unsigned (&y)[7], unsigned& sg) {
  unsigned a[4], b[4];
  any_words(va, A, a);
  any_words(vb, A, b);
  sg = sign2(va, vb).mul;
  y[0] = __byte_perm(a[3], b[3], 0x5410);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    y[1 + 2 * j] = __byte_perm(a[2 - j], b[2 - j], 0x7632);
    y[2 + 2 * j] = __byte_perm(a[2 - j], b[2 - j], 0x5410);
  }
}
// Group G of any values from their lane words: slabs 5 G .. min(5 G + 4, 13).
template <int G, int W>
__device__ __forceinline__ void store_any(unsigned dst, unsigned slab_bytes, const unsigned (&y)[W / 2][7],
                                          const unsigned (&sg)[W / 2], unsigned e1024) {
#pragma unroll
  for (int j = 0; j < kGroup; ++j) {
    const int s = G * kGroup + j;
    if (s >= kAll) break;
    unsigned w[W / 2];
#pragma unroll
    for (int m = 0; m < W / 2; ++m) {
      const Sign2 f{sg[m], hmul2(sg[m], s == 0 ? 0xE400E400u : 0xE480E480u)};
      w[m] = s % 2 == 0 ? digit_hi(y[m][s / 2], e1024, f) : digit_lo(y[m][s / 2], e1024, f);
    }
    st_slab<W>(dst + (unsigned)j * slab_bytes, w);
  }
}
// A tile with all digits, 16 values (v) a thread: their lane words would not fit
// the registers, so they are cut eight at a time, groups 0 and 1 together once
// both buffers are free (the MMAs of groups G - 2 and G - 1 done), and the lowest
// words are kept for group 2 (store_any16_last, after the previous tile's
// epilogue, which covers group 0's MMAs).  Out of line, waits and arrivals included.
__device__ __noinline__ void store_any16(const double* v, int A, unsigned dst, unsigned slab_bytes, unsigned fb0,
                                         unsigned rb0, int G, volatile int* bad, unsigned* keep) {
  const unsigned e1024 = exp1024x2();
  const unsigned b = G & 1, buffer = kGroup * slab_bytes;
  if (G >= 2) {
    mbar_wait(fb0 + 8u * b, (unsigned)((G - 2) >> 1) & 1u, bad);
    mbar_wait(fb0 + 8u * (b ^ 1u), (unsigned)((G - 1) >> 1) & 1u, bad);
  }
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    unsigned y[4][7], sg[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      any_lanes(v[8 * h + 2 * m], v[8 * h + 2 * m + 1], A, y[m], sg[m]);
      keep[(4 * h + m) * 3] = y[m][5];
      keep[(4 * h + m) * 3 + 1] = y[m][6];
      keep[(4 * h + m) * 3 + 2] = sg[m];
    }
    const unsigned at = dst + (unsigned)h * 128u;
    store_any<0, 8>(at + b * buffer, slab_bytes, y, sg, e1024);
    store_any<1, 8>(at + (b ^ 1u) * buffer, slab_bytes, y, sg, e1024);
  }
  fence_proxy_async();
  mbar_arrive(rb0 + 8u * b);
  mbar_arrive(rb0 + 8u * (b ^ 1u));
}
// Group 2 of the tile whose group 0 was G.
__device__ __noinline__ void store_any16_last(const unsigned* keep, unsigned dst, unsigned slab_bytes, unsigned fb0,
                                              unsigned rb0, int G, volatile int* bad) {
  const unsigned e1024 = exp1024x2();
  const unsigned b = G & 1, buffer = kGroup * slab_bytes;
  mbar_wait(fb0 + 8u * b, (unsigned)(G >> 1) & 1u, bad);  // group 0's MMAs
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    unsigned y[4][7], sg[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      y[m][5] = keep[(4 * h + m) * 3];
      y[m][6] = keep[(4 * h + m) * 3 + 1];
      sg[m] = keep[(4 * h + m) * 3 + 2];
    }
    store_any<2, 8>(dst + (unsigned)h * 128u + b * buffer, slab_bytes, y, sg, e1024);
  }
  fence_proxy_async();
  mbar_arrive(rb0 + 8u * b);
}

// x 2^(1132 - A) as a signed 128-bit integer, truncated toward zero.
__device__ __forceinline__ i128 fixed_trunc(double x, int A) {
  const unsigned hi = hi32(x), lo = lo32(x);
  int be = (hi >> 20) & 0x7ff;
  unsigned mh = hi & 0xfffffu;
  if (be) mh |= 0x100000u; else be = 1;
  const unsigned long long m = ((unsigned long long)mh << 32) | lo;
  const int t = 57 - (A - be);
  u128 X;
  if (t >= 0) X = (u128)m << t;
  else if (t > -64) X = (u128)(m >> (-t));
  else X = 0;
  return (hi >> 31) ? -(i128)X : (i128)X;
}

// Outputs of a thread rounded side by side: one at a time where the next
// tile's values stand in registers meanwhile (kin = 64).
template <int W>
constexpr int kRoundSide = W >= 16 ? 1 : 4;
// Added to the exponent of a row or a column with a non-finite value (FP32 rows:
// of one that plain_rows takes), and to a row's when a wait has run out: no lean
// rounding takes it, and the general one answers NaN.
constexpr int kNaNExp = 1 << 24;
// The general exact rounding (rare inputs the lean forms leave),
// kept out of line so that the kernels' code stays small.
__device__ __noinline__ float round_general_f32(i128 h, int S) {
  return S >= kNaNExp / 2 ? __int_as_float(0x7fc00000) : w_to_float(h, S);
}
__device__ __noinline__ double round_general(bool update, double y, i128 h, int S) {
  if (S >= kNaNExp / 2) return __longlong_as_double(0x7ff8000000000000ll);
  bool ok;
  const double o = update ? w_to_double_fast(h, S, ok) : sub_round_fast(y, h, S, ok);
  if (ok) return o;
  return update ? w_to_double(h, S) : sub_round(y, h, S);
}

// FP32: binades between the largest entries of Z's rows beyond which all rows go
// through plain_rows.  Z = R^{-1} or M^{-1/2} of X = U D (columns of norm 1 times
// their norms d_i) has rows of about 1 / d_i, times at most kappa(U) < 2^27 (the
// largest that an FP64 Cholesky takes), while a digit sum is off by up to 2^-98
// max_i |x_ri| max_i |z_ij| <= 2^-98 max d max_i |z_ij| <= 2^(40 + 27 - 98) of a column
// of norm 1: below the FP32 rounding, and 2^-57 of it for a well-conditioned U.
constexpr int kUneven = 40;

// FP32 rows that the digits do not hold (k <= KM), summed in FP64 as update.cu
// does: the four lanes of a row (cg) read all of it before one of them stores, and
// take every fourth output.  Called by whole warps; rare, so out of line.
template <int KM, bool TRI>
__device__ __noinline__ void plain_rows(int k, const float* A, int64_t lda, const double* __restrict__ B, int ldb,
                                        float* Out, int64_t ldo, int cg, bool mine) {
  double x[KM];
#pragma unroll
  for (int i = 0; i < KM; ++i) x[i] = mine && i < k ? (double)A[(size_t)i * lda] : 0.0;
  __syncwarp();
  if (!mine) return;
#pragma unroll
  for (int j4 = 0; j4 < KM; j4 += 4) {
    const int j = j4 + cg;
    if (j >= k) break;
    const double* b = B + (size_t)j * ldb;
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < (TRI ? j4 + 4 : KM); ++i)
      if (TRI ? i <= j : i < k) s = __fma_rn(x[i], b[i], s);
    Out[(size_t)j * ldo] = (float)s;
  }
}

// KP = 4 W: the K dimension (kin padded to 16, 32 or 64; padded columns
// are converted as zeros).  KO: blocks of 16 output columns (1, or 2 for
// kout up to 32 with kin <= 32).  With one block, TMEM holds two
// accumulators and the epilogue of tile i - 1 overlaps the MMAs of tile i;
// with two, the 480 columns of the two blocks leave one accumulator each:
// the converters store groups 0 and 1 of tile i, read tile i - 1's
// accumulators, release them (tfree) and then store group 2, and the MMAs of
// tile i wait for that release, so the inputs are converted once for all 32
// outputs.
template <typename Real, bool UPDATE, int W, int KO>
__global__ void __launch_bounds__(kThreads, 1)
    umma_rowprod_kernel(int64_t n, int kin, const Real* A, int64_t lda, int kout,
                        const double* __restrict__ Bh, const double* __restrict__ Bl, int ldb, int tri,
                        const Real* Yin, int64_t ldyin, Real* Out, int64_t ldo, const int* gate) {
  if (gate && *gate == 0) return;
  constexpr int KP = 4 * W;
  constexpr int KC = KP / 16;             // MMAs (K = 16) per slab
  constexpr unsigned SBO = 16u * KP;      // bytes between 8-row groups of an operand
  constexpr unsigned SLAB_A = 16u * SBO;  // one digit slab of the tile (128 rows)
  constexpr unsigned B_BYTES = 2u * kAll * SBO;  // 14 slabs x 16 columns (one block of outputs)
  constexpr int NOUT = kOut * KO;
  static_assert(KO == 1 || (KO == 2 && W <= 8), "two output blocks only for kin <= 32");
  static_assert(std::is_same_v<Real, double> || (UPDATE && kStageValues<W>), "FP32: the update for kin <= 32");
  constexpr int NEAR = kNearOf<Real>;

  extern __shared__ __align__(128) unsigned char smem[];
  unsigned char* bdig = smem;                                  // the small matrix's digits
  unsigned char* adig = smem + KO * B_BYTES;                   // two group buffers of 5 slabs
  int* Arow = reinterpret_cast<int*>(adig + 2 * kGroup * SLAB_A);  // [2][128] row exponents
  int* Bexp = Arow + 2 * kRows;                                // [NOUT] column exponents
  Real* stg = reinterpret_cast<Real*>(Bexp + NOUT);            // [W][512] staged values (kin <= 32)
  __shared__ __align__(8) unsigned long long full_bar[2], ready_bar[2], tfree_bar;
  __shared__ unsigned tmem_base;
  __shared__ int bad;
  // FP32: the largest exponent of each row of the small matrix; whether it is too uneven for the digits
  [[maybe_unused]] __shared__ int zrow[32], uneven;
  __shared__ int far[2];  // far[i & 1] = i: the CTA's tile i needs all digits (set before the arrivals for its first group)

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t ntiles = (n + kRows - 1) / kRows;

  // ---- set-up: TMEM (two accumulators), barriers, the small matrix's digits
  if (warp == 0) tmem_alloc(smem_u32(&tmem_base), 2 * kAccCols);
  if (tid == 0) {
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&full_bar[b]), 1);
      mbar_init(smem_u32(&ready_bar[b]), kConvThreads);
    }
    mbar_init(smem_u32(&tfree_bar), kConvThreads);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    bad = 0;
    far[0] = far[1] = -1;
  }
  if constexpr (sizeof(Real) == 4) {
    if (tid < 32) zrow[tid] = 0;
    if (tid == 0) uneven = 0;
    __syncthreads();
  }
  // column exponents, a warp to a column (one round of loads: a thread to a
  // column, one load after another, made a launch of 64 x 16 10 us longer)
  for (int j = warp; j < NOUT; j += kThreads / 32) {
    int e = 0;
    bool nf = false;
    if (j < kout) {
      for (int i = lane; i < kin; i += 32) {
        if (tri && i > j) continue;
        const int ae = align_exp(Bh[(size_t)j * ldb + i]);
        e = max(e, ae);
        if constexpr (sizeof(Real) == 4) atomicMax(&zrow[i], ae);
        nf |= ae == 2047 || (Bl && align_exp(Bl[(size_t)j * ldb + i]) == 2047);
      }
    }
    e = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
    nf = __any_sync(0xffffffffu, nf);
    // one binade of headroom: |h + l| may round up past the largest h
    if (lane == 0) Bexp[j] = e + 1 + (nf ? kNaNExp : 0);
    if constexpr (sizeof(Real) == 4) {
      if (nf) uneven = 1;
    }
  }
  __syncthreads();
  if constexpr (sizeof(Real) == 4) {
    if (warp == 0) {
      const int e = lane < kin ? zrow[lane] : 0;
      const int hi = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
      const int lo = (int)__reduce_min_sync(0xffffffffu, e ? (unsigned)e : 4095u);
      if (lane == 0 && hi - lo > kUneven) uneven = 1;
    }
  }
  for (int e = tid; e < NOUT * KP; e += kThreads) {  // block j / 16: B row R = t * 16 + j % 16 (slab t), K index i
    const int j = e / KP, i = e % KP;
    i128 x = 0;
    if (j < kout && i < kin && !(tri && i > j) && Bexp[j] < kNaNExp) {
      const double h = Bh[(size_t)j * ldb + i], l = Bl ? Bl[(size_t)j * ldb + i] : 0.0;
      x = fixed_trunc(h, Bexp[j]) + fixed_trunc(l, Bexp[j]);
    }
    const bool neg = x < 0;
    const u128 U = (neg ? (u128)(-x) : (u128)x) + (((u128)0x8080808080ull << 64) | 0x8080808080808080ull);  // < 2^110 + bias
    for (int t = 0; t < kAll; ++t) {
      const int f = (int)((unsigned)(U >> (104 - 8 * t)) & 255u) - (t ? 128 : 0);
      const int R = t * kOut + j % kOut;
      *reinterpret_cast<__half*>(bdig + (j / kOut) * B_BYTES + (R >> 3) * SBO + (i >> 3) * 128 + (R & 7) * 16 +
                                 (i & 7) * 2) = __int2half_rn(neg ? -f : f);
    }
  }
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const unsigned taddr = tmem_base;
  const unsigned fb0 = smem_u32(&full_bar[0]), rb0 = smem_u32(&ready_bar[0]), tfb = smem_u32(&tfree_bar);
  const unsigned adig_s = smem_u32(adig), bdig_s = smem_u32(bdig);

  if (sizeof(Real) == 4 && uneven) {
    // ---------------- FP32, columns of X too uneven for the digits: every row in FP64
    if constexpr (sizeof(Real) == 4) {
      const int64_t r = (int64_t)warp * 8 + (lane & 7);
      for (int64_t T = blockIdx.x; T < ntiles && warp < kConvWarps; T += gridDim.x) {
        const int64_t gr = T * kRows + r;
        if (tri) plain_rows<KP, true>(kin, A + gr, lda, Bh, ldb, Out + gr, ldo, lane >> 3, gr < n);
        else plain_rows<KP, false>(kin, A + gr, lda, Bh, ldb, Out + gr, ldo, lane >> 3, gr < n);
      }
    }
  } else if (warp == kConvWarps) {
    // ---------------- MMA issuer
    if (lane == 0) {
      int G = 0;  // groups issued
      bool ok = true;
      for (int64_t T = blockIdx.x, i = 0; T < ntiles && ok; T += gridDim.x, ++i) {
        const unsigned acc = taddr + (KO > 1 ? 0u : (unsigned)(i & 1) * kAccCols);
        if constexpr (KO > 1) {
          if (i > 0) {  // tile i - 1's accumulators read by its epilogue
            if (!mbar_wait(tfb, (unsigned)(i - 1) & 1u, &bad)) break;
            tc_fence_after();
          }
        }
        int ng = kGroupsNear, nslabs = NEAR;
#pragma unroll 1
        for (int g = 0; g < ng; ++g, ++G) {
          const int b = G & 1;
          if (!mbar_wait(rb0 + 8u * b, (unsigned)(G >> 1) & 1u, &bad)) {
            ok = false;
            break;
          }
          if (g == 0 && *reinterpret_cast<volatile int*>(&far[i & 1]) == (int)i) ng = kGroupsAll, nslabs = kAll;
          tc_fence_after();
          const unsigned abuf = adig_s + (unsigned)b * kGroup * SLAB_A;
          const int ns = min(kGroup, nslabs - g * kGroup);
          for (int sg = 0; sg < ns; ++sg) {
            const int s = g * kGroup + sg;
            const unsigned idesc = idesc_f16(kRows, kOut * (kAll - s));
#pragma unroll
            for (int h = 0; h < KO; ++h)
#pragma unroll
              for (int kc = 0; kc < KC; ++kc) {
                const unsigned long long ad = sdesc(abuf + (unsigned)sg * SLAB_A + (unsigned)kc * 256u, 128u, SBO);
                const unsigned long long bd = sdesc(bdig_s + (unsigned)h * B_BYTES + (unsigned)kc * 256u, 128u, SBO);
                mma_f16(acc + (unsigned)h * kAccCols + (unsigned)(kOut * s), ad, bd, idesc,
                        (s == 0 && kc == 0) ? 0u : 1u);
              }
          }
          mma_commit(fb0 + 8u * b);
        }
      }
      // the last committed MMAs finish before TMEM and shared memory are released
      if (G > 0) mbar_wait_final(fb0 + 8u * ((G - 1) & 1), (unsigned)((G - 1) >> 1) & 1u, &bad);
    }
    __syncwarp();
  } else {
    // ---------------- converters: loads, row exponents, digits; epilogues
    const int rlo = lane & 7, cg = lane >> 3;
    const int r = warp * 8 + rlo;  // tile row of this thread's values
    const int c0 = cg * W;         // first of its W columns
    // digit offset of (row r, column c0) within a slab
    const unsigned dofs = (unsigned)(r >> 3) * SBO + (unsigned)(c0 >> 3) * 128u + (unsigned)(r & 7) * 16u +
                          (unsigned)(c0 & 7) * 2u;
    // epilogue mapping: TMEM lane quarter warp % 4; the kout outputs of a block
    // are dealt to the four warps of a quarter, ny = ceil(kout / 4) to each
    const int eq = warp & 3, ep = warp >> 2;
    const int L = eq * 32 + lane;
    const unsigned tq = taddr + ((unsigned)(eq * 32) << 16);

    // the values of tile T into this thread's staging slots (zeros beyond the
    // matrix: nothing is read there)
    const int nv = min(max(kin - c0, 0), W);  // columns of this thread
    const unsigned stg_s = smem_u32(stg) + (unsigned)(tid * sizeof(Real));
    auto prefetch = [&](int64_t T) {
      const int64_t gr = T * kRows + r;
      const int in = gr < n ? nv : 0;  // (T >= ntiles: gr >= n)
      const Real* src = A + (in > 0 ? (size_t)c0 * lda + gr : 0);
#pragma unroll
      for (int k = 0; k < W; ++k) {
        const unsigned dst = stg_s + (unsigned)(k * kConvThreads * sizeof(Real));
        if constexpr (sizeof(Real) == 8) cp_async8z(dst, src, k < in ? 8u : 0u);
        else cp_async4z(dst, src, k < in ? 4u : 0u);
        if (k + 1 < in) src += lda;
      }
      cp_async_commit_group();
    };
    if constexpr (kStageValues<W>) prefetch(blockIdx.x);

    // outputs j0 .. j0 + ny - 1 of this warp (output block ob) of tile T
    auto epilogue_ny = [&](auto NYc, int64_t T, int64_t i, int ob) {
      constexpr int ny = decltype(NYc)::value;
      const int j0 = ob * kOut + ep * ny;
      if (j0 >= kout) return;  // all outputs of this warp are padding (warp-uniform)
      const unsigned tb = tq + (unsigned)(KO > 1 ? ob : (int)(i & 1)) * kAccCols + (unsigned)(ep * ny);
      // (FP32: a row of plain_rows stands beyond the matrix)
      const int64_t grow = sizeof(Real) == 4 && Arow[(i & 1) * kRows + L] >= kNaNExp ? n : T * kRows + L;
      double yv[ny];
      {
        const Real* Yp = Yin + (size_t)j0 * ldyin + grow;
#pragma unroll
        for (int y = 0; y < ny; ++y)
          yv[y] = (!UPDATE && j0 + y < kout && grow < n) ? Yp[(size_t)y * ldyin] : 0.0;
      }
      // pairs q_m = S_2m 256 + S_2m+1 + kPairOffset (m = 0..6) in 32 bits;
      // h + kOffset = sum_m q_m 2^(16 (6 - m)): the even pairs are its words, the
      // odd ones lie half a word up
      u128 h[ny];
      {
        unsigned q[ny][7];
        float squares[ny] = {};
        // (two buffers of loads cost the kin = 64 kernel more spills than they hide)
        constexpr int kBuf = W < 16 ? 2 : 1;
        unsigned v[kBuf][4][4], vl[2][4];
        auto pairs = [&](int m, const unsigned(&a)[4], const unsigned(&b)[4]) {
#pragma unroll
          for (int y = 0; y < ny; ++y) {
            const float fa = __uint_as_float(a[y]), fb = __uint_as_float(b[y]);
            q[y][m] = __float_as_uint(fa + 0x1.8p23f) * 256u + __float_as_uint(fb + 0x1.8p23f);
            if constexpr (!kSmallDiag<W>) squares[y] = fmaf(fa, fa, fmaf(fb, fb, squares[y]));
          }
        };
        tmem_ld4(tb, v[0]);
        tmem_wait4(v[0]);
#pragma unroll
        for (int t = 0; t < 3; ++t) {  // diagonals 4 t .. 4 t + 3
          auto next = [&]() {
            if (t < 2) tmem_ld4(tb + (unsigned)((4 * t + 4) * kOut), v[(t + 1) % kBuf]);
            else tmem_ld4(tb + (unsigned)(12 * kOut), vl);
          };
          if (kBuf > 1) next();
          pairs(2 * t, v[t % kBuf][0], v[t % kBuf][1]);
          pairs(2 * t + 1, v[t % kBuf][2], v[t % kBuf][3]);
          if (kBuf == 1) next();
          if (t < 2) tmem_wait4(v[(t + 1) % kBuf]);
          else tmem_wait4(vl);
        }
        pairs(6, vl[0], vl[1]);
        float most = 0.f;
#pragma unroll
        for (int y = 0; y < ny; ++y) {
          h[y] = pairs_sum(q[y]);
          most = fmaxf(most, squares[y]);
        }
        if constexpr (!kSmallDiag<W>) {
          if (__any_sync(0xffffffffu, most >= kSquares)) {
            u128 g[4];
            combine_any(tb, g);
#pragma unroll
            for (int y = 0; y < ny; ++y) h[y] = g[y];
          }
        }
      }
      const int Sr = Arow[(i & 1) * kRows + L] - kScaleProd + (bad ? kNaNExp : 0);
      Real* Op = Out + (size_t)j0 * ldo + grow;
      // the roundings of kSide outputs side by side (no branches among them);
      // what they do not take is rounded by the general functions
      constexpr int kSide = kRoundSide<W> < ny ? kRoundSide<W> : ny;
#pragma unroll
      for (int y0 = 0; y0 < ny; y0 += kSide) {
        Real o[kSide];
        unsigned left = 0;
        auto round_side = [&](auto FAR) {
#pragma unroll
          for (int y = y0; y < y0 + kSide && y < ny; ++y) {
            const int S = Sr + Bexp[j0 + y];
            bool ok;
            if constexpr (!UPDATE) o[y - y0] = sub_round_lean<decltype(FAR)::value>(yv[y], h[y], kOffset, S, ok);
            else if constexpr (sizeof(Real) == 8) o[y - y0] = w_to_double_lean(h[y] - kOffset, S, 0u, ok);
            else o[y - y0] = w_to_float_lean(h[y] - kOffset, S, ok);
            left |= ok || j0 + y >= kout || grow >= n ? 0u : 1u << y;
          }
        };
        bool far_y = false;
        if constexpr (!UPDATE) {
#pragma unroll
          for (int y = y0; y < y0 + kSide && y < ny; ++y) far_y |= dominates(yv[y], Sr + Bexp[j0 + y]);
        }
        if (!UPDATE && __any_sync(0xffffffffu, far_y)) round_side(std::true_type{});
        else round_side(std::false_type{});
        if (__any_sync(0xffffffffu, left != 0u)) {
          u128 g[4];  // formed anew when several outputs' sums would have to be kept
          if constexpr (kSide > 1) combine_any(tb, g);
#pragma unroll
          for (int y = y0; y < y0 + kSide && y < ny; ++y) {
            if constexpr (kSide == 1) g[y] = h[y];
            if (left >> y & 1u) {
              const i128 w = (i128)(g[y] - kOffset);
              const int S = Sr + Bexp[j0 + y];
              if constexpr (sizeof(Real) == 4) o[y - y0] = round_general_f32(w, S);
              else o[y - y0] = round_general(UPDATE, UPDATE ? 0.0 : Yin[(size_t)(j0 + y) * ldyin + grow], w, S);
            }
          }
        }
#pragma unroll
        for (int y = y0; y < y0 + kSide && y < ny; ++y)
          if (grow < n && j0 + y < kout) Op[(size_t)y * ldo] = o[y - y0];
      }
    };
    auto epilogue_block = [&](int64_t T, int64_t i, int ob) {
      switch (min((kout - ob * kOut + 3) >> 2, 4)) {
        case 1: epilogue_ny(std::integral_constant<int, 1>{}, T, i, ob); break;
        case 2: epilogue_ny(std::integral_constant<int, 2>{}, T, i, ob); break;
        case 3: epilogue_ny(std::integral_constant<int, 3>{}, T, i, ob); break;
        default: epilogue_ny(std::integral_constant<int, 4>{}, T, i, ob); break;
      }
    };

    // this thread's W values of row r of tile T (zero beyond the matrix)
    auto load_direct = [&](int64_t T, double (&v)[W]) {
      const int64_t gr = T * kRows + r;
      const int in = gr < n ? nv : 0;
      const Real* src = A + (size_t)c0 * lda + gr;
#pragma unroll
      for (int k = 0; k < W; ++k) v[k] = k < in ? src[(size_t)k * lda] : 0.0;
    };
    double v[W];  // the values of the tile to come
    // takes the staged values of the tile that prefetch was last called for
    auto take = [&]() {
      asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll
      for (int k = 0; k < W; ++k) {
        if constexpr (sizeof(Real) == 8) v[k] = stg[k * kConvThreads + tid];
        else v[k] = widen(stg[k * kConvThreads + tid]);
      }
    };
    // The row's exponent: max of the |x| high words over the four threads of
    // the row (a row of subnormals and zeros has exponent field 0 and is aligned
    // to 1, the subnormals' own exponent); whether this thread's values hold a
    // zero; whether one of them is nonzero and below the near window.
    int Ar = 1;
    bool nonfinite = false, zeros = false;
    auto look = [&]() -> bool {
      unsigned key = 0, low = 0xffffffffu;
#pragma unroll
      for (int k = 0; k < W; ++k) {
        key = max(key, abs_hi(v[k]));
        low = min(low, abs_hi(v[k]));
      }
      key = max(key, __shfl_xor_sync(0xffffffffu, key, 8));
      key = max(key, __shfl_xor_sync(0xffffffffu, key, 16));
      const int e = (int)(key >> 20);
      Ar = max(e, 1);
      nonfinite = e == 2047;
      const unsigned floor = near_floor(Ar);
      bool below = false;
      zeros = __any_sync(0xffffffffu, low < floor);
      if (zeros) {
#pragma unroll
        for (int k = 0; k < W; ++k) below |= abs_hi(v[k]) < floor && (abs_hi(v[k]) | lo32(v[k])) != 0u;
      }
      if constexpr (sizeof(Real) == 4) below |= nonfinite;  // (looked at again where all digits are cut)
      return below;
    };
    const unsigned e1024 = exp1024x2();
    bool all = false;  // the tile to come needs all digits
    {
      bool below;
      if constexpr (kStageValues<W>) {
        take();
        below = look();
        prefetch(blockIdx.x + (int64_t)gridDim.x);
      } else {
        load_direct(blockIdx.x, v);
        below = look();
      }
      all = bar_conv_or<kConvThreads>(below);
    }

    int G = 0;
    int64_t Tprev = -1, iprev = 0;
    for (int64_t T = blockIdx.x, i = 0; T < ntiles; T += gridDim.x, ++i) {
      if (cg == 0) {
        Arow[(i & 1) * kRows + r] = Ar + (nonfinite && sizeof(Real) == 8 ? kNaNExp : 0);
      }
      if (all && tid == 0) *reinterpret_cast<volatile int*>(&far[i & 1]) = (int)i;
      const int ng = all ? kGroupsAll : kGroupsNear;
      unsigned z[W / 2][5], sg[W / 2];
      [[maybe_unused]] unsigned keep[24];  // (kin = 64, all digits: for group 2)
      if (!all) {
        if (zeros) near_lanes<W, true>(v, Ar, z, sg);
        else near_lanes<W, false>(v, Ar, z, sg);
      }
      // groups of slabs into the alternating buffers
      auto group = [&](int g, auto store) {
        const int b = G & 1;
        if constexpr (KO > 1) {
          if (g == ng - 1 && Tprev >= 0) {
            // one accumulator per output block: the previous tile's epilogue
            // reads them here and releases them to this tile's MMAs (which are
            // not issued before, so no group of this tile may be waited for).
            // The previous tile's last group is G - 2 at a tile's second group:
            // waited for here, or before this tile's second group was stored
            if (g == 1) mbar_wait(fb0 + 8u * b, (unsigned)((G - 2) >> 1) & 1u, &bad);
            tc_fence_after();
#pragma unroll 1
            for (int ob = 0; ob < KO; ++ob) epilogue_block(Tprev, iprev, ob);
            tc_fence_before();
            mbar_arrive(tfb);
          }
        }
        if (G >= 2) mbar_wait(fb0 + 8u * b, (unsigned)((G - 2) >> 1) & 1u, &bad);  // MMAs of group G - 2 done
        store(adig_s + (unsigned)b * kGroup * SLAB_A + dofs);
        fence_proxy_async();
        mbar_arrive(rb0 + 8u * b);
        ++G;
      };
      if (!all) {
        group(0, [&](unsigned dst) { store_near<0, kGroup, W>(dst, SLAB_A, z, sg, e1024); });
        group(1, [&](unsigned dst) { store_near<1, NEAR - kGroup, W>(dst, SLAB_A, z, sg, e1024); });
      } else if constexpr (W <= 8) {
        unsigned y[W / 2][7];
        [[maybe_unused]] bool plain = false;  // FP32: the row goes through plain_rows
        if constexpr (sizeof(Real) == 4) {
          // (24 bits that begin more than 86 binades below the row's largest reach
          // below the digits' last bit)
          const unsigned last = (unsigned)max(Ar - 86, 0) << 20;
#pragma unroll
          for (int k = 0; k < W; ++k) plain |= abs_hi(v[k]) < last && abs_hi(v[k]) != 0u;
          plain |= __shfl_xor_sync(0xffffffffu, plain, 8);
          plain |= __shfl_xor_sync(0xffffffffu, plain, 16);
          plain |= nonfinite;
        }
#pragma unroll
        for (int m = 0; m < W / 2; ++m) any_lanes(v[2 * m], v[2 * m + 1], Ar, y[m], sg[m]);
#pragma unroll 1
        for (int g = 0; g < kGroupsAll; ++g)
          group(g, [&](unsigned dst) {
            if (g == 0) store_any<0, W>(dst, SLAB_A, y, sg, e1024);
            else if (g == 1) store_any<1, W>(dst, SLAB_A, y, sg, e1024);
            else store_any<2, W>(dst, SLAB_A, y, sg, e1024);
          });
        if constexpr (sizeof(Real) == 4) {
          // (the tile's values stand in memory until its epilogue, which passes these rows over)
          if (__any_sync(0xffffffffu, plain)) {
            const int64_t gr = T * kRows + r;
            if (tri) plain_rows<KP, true>(kin, A + gr, lda, Bh, ldb, Out + gr, ldo, cg, plain && gr < n);
            else plain_rows<KP, false>(kin, A + gr, lda, Bh, ldb, Out + gr, ldo, cg, plain && gr < n);
            if (plain && cg == 0) Arow[(i & 1) * kRows + r] = Ar + kNaNExp;
          }
        }
      } else {
        double u[W];
#pragma unroll
        for (int k = 0; k < W; ++k) u[k] = v[k];
        store_any16(u, Ar, adig_s + dofs, SLAB_A, fb0, rb0, G, &bad, keep);
        G += kGroupsAll;
      }
      // the next tile's values: in flight during the epilogue
      if constexpr (!kStageValues<W>) load_direct(T + gridDim.x, v);
      if (!UPDATE && tid < 8 * kout) {  // Y of this tile, read by its epilogue a tile from now: into L2
        const int64_t g0 = T * kRows + (tid & 7) * 16;  // 16 rows = one 128-byte line per thread
        if (g0 < n) prefetch_l2(Yin + (size_t)(tid >> 3) * ldyin + g0);
      }
      // the previous tile's MMAs completed (all but its last group were waited
      // for before this tile's groups were written, the last one here): its
      // epilogue overlaps this tile's MMAs
      if constexpr (KO == 1) {
        if (Tprev >= 0) {
          tc_fence_after();
          epilogue_block(Tprev, iprev, 0);
          tc_fence_before();
        }
      }
      if constexpr (W > 8) {
        if (all) store_any16_last(keep, adig_s + dofs, SLAB_A, fb0, rb0, G - kGroupsAll, &bad);
      }
      bool below;
      if constexpr (kStageValues<W>) {
        take();
        below = look();  // (reads every value before their slots are refilled)
        prefetch(T + 2 * (int64_t)gridDim.x);
      } else {
        below = look();
      }
      // every warp has read buffer (i - 1) & 1 of the row exponents, and the
      // next tile's kind is agreed on
      all = bar_conv_or<kConvThreads>(below);
      Tprev = T;
      iprev = i;
    }
    if (Tprev >= 0) {  // the last tile
      mbar_wait(fb0 + 8u * ((G - 1) & 1), (unsigned)((G - 1) >> 1) & 1u, &bad);
      tc_fence_after();
      if constexpr (KO == 1) {
        epilogue_block(Tprev, iprev, 0);
      } else {
#pragma unroll 1
        for (int ob = 0; ob < KO; ++ob) epilogue_block(Tprev, iprev, ob);
      }
      tc_fence_before();
    }
    if constexpr (kStageValues<W>) asm volatile("cp.async.wait_all;" ::: "memory");  // the last (empty) prefetch
  }

  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(taddr, 2 * kAccCols);
  }
}

template <int W, int KO>
size_t smem_bytes() {
  constexpr int KP = 4 * W;
  const size_t sbo = 16u * KP;
  const size_t b = KO * 2 * kAll * sbo, a = 2 * kGroup * 16 * sbo, small = (2 * kRows + kOut * KO) * sizeof(int);
  const size_t stage = kStageValues<W> ? (size_t)W * kConvThreads * sizeof(double) : 0;
  return std::max(b + a + small + stage, kMinSmem);
}

template <typename Real, bool UPDATE, int W, int KO>
cudaError_t launch_w(int64_t n, int kin, const Real* A, int64_t lda, int kout, const double* Bh, const double* Bl,
                     int ldb, bool tri, const Real* Yin, int64_t ldyin, Real* Out, int64_t ldo, const int* gate,
                     cudaStream_t st, int ctas) {
  const size_t smem = smem_bytes<W, KO>();
  cudaError_t e = set_dyn_smem(umma_rowprod_kernel<Real, UPDATE, W, KO>, smem);
  if (e != cudaSuccess) return e;
  const int64_t ntiles = (n + kRows - 1) / kRows;
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(ntiles, ctas > 0 ? ctas : 152));
  umma_rowprod_kernel<Real, UPDATE, W, KO><<<grid, kThreads, smem, st>>>(n, kin, A, lda, kout, Bh, Bl, ldb, tri ? 1 : 0,
                                                                      Yin, ldyin, Out, ldo, gate);
  return cudaGetLastError();
}

template <bool UPDATE>
cudaError_t launch_mode(int64_t n, int kin, const double* A, int64_t lda, int kout, const double* Bh, const double* Bl,
                        int ldb, bool tri, const double* Yin, int64_t ldyin, double* Out, int64_t ldo, const int* gate,
                        cudaStream_t st, int ctas) {
  if (kout > kOut)  // two blocks of output columns (kin <= 32): the inputs converted once
    return launch_w<double, UPDATE, 8, 2>(n, kin, A, lda, kout, Bh, Bl, ldb, tri, Yin, ldyin, Out, ldo, gate, st, ctas);
  if (kin <= 16)
    return launch_w<double, UPDATE, 4, 1>(n, kin, A, lda, kout, Bh, Bl, ldb, tri, Yin, ldyin, Out, ldo, gate, st, ctas);
  if (kin <= 32)
    return launch_w<double, UPDATE, 8, 1>(n, kin, A, lda, kout, Bh, Bl, ldb, tri, Yin, ldyin, Out, ldo, gate, st, ctas);
  return launch_w<double, UPDATE, 16, 1>(n, kin, A, lda, kout, Bh, Bl, ldb, tri, Yin, ldyin, Out, ldo, gate, st, ctas);
}

}  // namespace

cudaError_t umma_rowprod_take_wait_record(unsigned* out) { return take_wait_record(out); }

bool umma_rowprod_supported(int64_t n, int kin, int kout) {
  const char* e = getenv("EO_DD_ROW_ENGINE");
  if (e && e[0] == 'i') return false;
  if (kin < 1 || kin > 64 || kout < 1 || kout > 2 * kOut || (kout > kOut && kin > 32)) return false;
  if (e && e[0] == 'u') return true;  // (for comparisons: the tensor cores wherever they can run)
  // Small products run faster on the integer limbs, whose cost follows
  // kin kout, while a tile here costs its digits and at least one output for
  // every warp.  Measured, integer limbs vs tiles: on 1e6 rows 4 x 4 68 vs
  // 111 us, 8 x 4 105 vs 120, 10 x 4 163 vs 121, 8 x 8 205 vs 139, 16 x 8 336
  // vs 139, 16 x 16 587 vs 177.  Rows of up to 8 entries stay in the
  // registers of a thread there, which starts quicker: 8 x 8 on 1e4 rows 8.3
  // vs 10.3 us, equal on 2e4, on 4e4 16.5 vs 14.4 (16 x 4, 2e3 rows: 12.4 vs 10.3).
  const int entries = kin * std::max(kout, 4);
  return entries >= 128 || (entries >= 40 && (kin > 8 || n >= 32768));
}

cudaError_t launch_umma_rowprod(bool update, int64_t n, int kin, const double* A, int64_t lda, int kout,
                                const double* Bh, const double* Bl, int ldb, bool tri, const double* Yin,
                                int64_t ldyin, double* Out, int64_t ldo, const int* gate, cudaStream_t st,
                                int ctas) {
  if (n <= 0) return cudaSuccess;
  return update ? launch_mode<true>(n, kin, A, lda, kout, Bh, Bl, ldb, tri, Yin, ldyin, Out, ldo, gate, st, ctas)
                : launch_mode<false>(n, kin, A, lda, kout, Bh, Bl, ldb, tri, Yin, ldyin, Out, ldo, gate, st, ctas);
}

cudaError_t launch_umma_update_f32(int64_t n, int k, float* X, int64_t ldx, const double* Zh, const double* Zl, int ldz,
                                   bool tri, const int* gate, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const float* none = nullptr;
  if (k > kOut) return launch_w<float, true, 8, 2>(n, k, X, ldx, k, Zh, Zl, ldz, tri, none, 0, X, ldx, gate, st, 0);
  return launch_w<float, true, 4, 1>(n, k, X, ldx, k, Zh, Zl, ldz, tri, none, 0, X, ldx, gate, st, 0);
}

}  // namespace eo
