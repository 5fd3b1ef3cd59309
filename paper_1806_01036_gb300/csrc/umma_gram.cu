// umma_gram.cu — compensated Gram products G = X^T Y on the 5th-generation
// tensor cores (tcgen05.mma, accumulators in tensor memory).
//
// arXiv:1806.01036, Sec. 4.2: M = Y~^T Y~ and W^T X summed over n rows with
// increased precision.  The sums are exact, as in fx.cuh; the digit products
// run on the tensor cores:
//
//  * each value x of a column is aligned to the column's alignment exponent
//    A and held as X = floor(|x| 2^(1132 - A)) < 2^110, written with 14
//    balanced base-256 digits, X = sum_s D_s 2^(104 - 8s), D_s in [-128, 127]
//    (D_0 in [0, 64]; the fields of X + sum_s 128 2^(104 - 8s), less 128);
//  * a digit is the FP16 integer sign(x) D_s, so a product of two digits is
//    an integer of at most 2^14 and FP32 sums of up to 1024 such products are
//    exact;
//  * a value within 25 binades of A has digits 10..13 zero (its X has a zero
//    low word); panels whose values all are such ("near", nearly always)
//    store and multiply only ten digit slabs;
//  * a column's alignment exponent starts at the first panel's largest
//    exponent plus EO_GRAM_HEADROOM binades and grows (to the new largest
//    exponent plus the headroom) only when a value's exponent exceeds it:
//    with the headroom, later panels rarely raise it, and each raise costs a
//    full drain of the accumulators;
//  * digit slabs sit in shared memory in the canonical K-major layout (8x16-
//    byte core matrices; the K dimension is the row index of X and Y).  One
//    MMA multiplies J consecutive X slabs (M = 128 = J x kxp TMEM lanes) by
//    the Y slabs t = 0 .. T-1 (N = T x kyp) and writes at TMEM column offset
//    J q kyp, so the product of slabs s = Jq + j and t lands in column block
//    c = Jq + t of lane block j: column block c of lane block j collects the
//    digit diagonal d = c + j; pairs with d > 14 are dropped;
//  * a symmetric 16-column product needs one MMA per 16 rows (q = 0): with
//    U(i, j) the sum of its column blocks c <= 7 and V(i, j) that of c >= 8
//    (s <= 7, t >= 8), the pairs with s >= 8 are those of V transposed, and
//    G(i, j) = U(i, j) + V(i, j) + V(j, i);
//  * before an accumulator can exceed 2^24 in magnitude (group_pairs below)
//    the accumulators are read back (tcgen05.ld), converted to integers,
//    added to 32-bit running sums per (lane, column) kept in TMEM and set
//    back to zero.  The running sums are folded into 128-bit totals every
//    kFoldDrains drains, before an alignment exponent grows, and at the end.  A
//    fold drops only the bits that the sum of the chunk's rows could push out of
//    127 (fold_bits: 5 for 132 rows, 13 for 26,000, 20 for the 2^22 of the
//    largest chunk; of all parts' rows when parts are added up): the unit is
//    2^(Ax + Ay - 2168 + drop).  The row-chunk partials go through the same exact,
//    order-free reduction (fx_gram_reduce).
//
// Error per product x y: the dropped digit pairs (d >= 15, twelve of weight
// 2^88 and fewer of smaller weights, each product at most 2^14) sum to less
// than 2^105.7 units^2 (units of 2^(Ax - 1132), 2^(Ay - 1132)), and a value
// more than 57 binades below A is truncated by less than one unit, which with
// max|x| >= 2^(109 - h) units for a headroom h is 2^(h - 109) max|x| max|y| of a
// product.  Together, with the same for y: below 2^-105.7 max|x| max|y| (h = 2).
// A fold rounds a lane's sum down by less than a unit, 2^(drop - 118) max|x|
// max|y|, and an entry of a symmetric tile adds 24 lanes: spread over the rows
// 2^-114 a product, and on the longest chunks, which fold many times, 2^-108.
// (Always dropping 20 bits was off by 2^-96.2 on two rows; keeping them
// in a word of its own per lane made a product of few rows 14.6 -> 17.5 us.)
//
// Pipeline per CTA (one per SM, 16 warps of 128 registers): the values of a
// panel of P rows arrive by TMA (two panels ahead, 16-row boxes with 128-byte
// swizzle).  A converter thread owns eight consecutive rows of one column of
// every panel, so that its column's alignment exponent stays in a register and
// its digits of a slab are one 16-byte shared-memory store (one row of a core
// matrix: eight lanes fill one, no bank conflicts).  Per panel it cuts its
// values as if they were near, takes the next panel's values from the staging
// buffer and looks whether they are (one unsigned range test), and, once every
// warp has stored the previous panel, stores its digits into the buffer that
// the MMAs of two panels ago have released, drains its share of the
// accumulators when due, and arrives; the sixteenth warp then issues the
// panel's MMAs and the copies of the panel after the next.  A warp that holds a
// zero masks it (4e6 x 64 + 16 with a zero column 1.04 ms, with every tenth value
// zero 1.04, dense 1.02).  A panel that holds a value other than zero below the
// near window is stored and multiplied with all 14 slabs, in steps that fit the
// digit buffers; only the warps that hold such values cut the last four digits,
// in a branch of its own, the others store zeros.  (One value in 100,000 / 10,000
// / 1,000 below it: 1.07 / 1.30 / 1.79 ms; through barriers, a second read and a
// second conversion of the panel by every warp, as a growth takes it, 1.13 / 1.80 /
// 3.40; 15 7-bit slabs of a panel in one buffer took 1.42 / 1.43 / 1.51.)  A value
// above its column's exponent sends every warp through a branch with barriers in
// which the exponents grow.  Every wait is
// bounded; a wait that runs out marks the partials non-finite, so the result
// is NaN.  Operands that TMA cannot address (a base not 16-byte aligned, an
// odd leading dimension, FP32) are copied by the converter threads with
// cp.async into the same places.
//
// What bounds it: issue and latency of the digit conversion (ALU pipe 48 % of
// active cycles, issue 51 %, tensor pipe 29 %, shared-memory data pipe 56 % of
// its wavefronts), not DRAM (30 %).  8-bit digits cost two ALU operations per
// pair of values and two digits (a byte permutation, or a masked merge, and an
// f16x2 FMA on the other pipe each) where 7-bit digits took three, and ten
// stored slabs instead of fifteen.  Measured, 4e6 rows against the 7-bit form
// (15 slabs, items of two rows, 19 converter warps): V^T Y 64 x 16 1.41 -> 1.04
// ms (2.5 TB/s), X^T X 16 columns 0.395 -> 0.264, 64 columns (strips) 4.6 ->
// 3.06.  Tried and slower: loads straight into registers (each 128-bit load
// costs 20 wavefronts of the shared data pipe: 1.30 ms), one bulk copy per
// column (80 a panel: 2.41 ms), four warps that only drain (each drain takes
// one of them 3,600 cycles, which the MMAs wait for: 1.08 ms), a barrier per
// panel over all warps (1.20 ms).
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstdlib>
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "fx.cuh"
#include "umma.cuh"

namespace eo {
namespace {

using namespace fx;
using namespace umma;

constexpr int kConvWarps = 15;              // convert
constexpr int kWarps = kConvWarps + 1;      // all drain TMEM (4 per lane quarter); the last issues MMAs and copies
constexpr int kThreads = 32 * kWarps;
constexpr int kIssuer = 32 * kConvWarps;    // the thread that issues the MMAs
constexpr int kLanes = 128;                   // MMA M = TMEM lanes
constexpr int kDiag = 14;                     // last digit diagonal kept
constexpr int kOffsetDigits = 2168;  // value of h: h 2^(Ax + Ay - 2168)
// Running sums grow by at most 2^24 per drain: exact in 32 bits for 127.
constexpr int kFoldDrains = 96;
constexpr int kPairRows = 1024;  // digit products of magnitude <= 2^14 that an FP32 accumulator holds exactly
constexpr size_t kSmemCap = 225 * 1024;
// Binades of headroom above a column's largest exponent when its alignment
// exponent is set (see the error bound above).
#ifndef EO_GRAM_HEADROOM
#define EO_GRAM_HEADROOM 2
#endif

// Digit pairs per row that a column block of any lane block collects at most,
// with ns digits per value: pairs (s, t) = (J q + j, c - J q), all < ns.
constexpr int group_pairs(int J, int ns, int nq) {
  int worst = 0;
  for (int c = 0; c <= kDiag; ++c)
    for (int j = 0; j < J; ++j) {
      int b = 0;
      for (int q = 0; q < nq; ++q)
        if (J * q + j < ns && c - J * q >= 0 && c - J * q < ns) ++b;
      worst = b > worst ? b : worst;
    }
  return worst;
}

// Geometry of one tile: KXP X columns by KYP Y columns; SHARED: Y = X (one
// operand held, 16 columns).  A warp converts 16 columns by 16 rows.
template <int KXP_, int KYP_, bool SHARED_>
struct Geo {
  static constexpr int KXP = KXP_, KYP = KYP_;
  static constexpr bool SHARED = SHARED_;
  static constexpr int COLS = KXP + (SHARED ? 0 : KYP);             // columns held
  static constexpr int NCG = (COLS + 15) / 16;                      // groups of 16 columns
  static constexpr int J = kLanes / KXP;                            // X slabs per MMA
  static constexpr int NQN = SHARED ? 1 : (kNear + J - 1) / J;      // MMAs per 16 rows, near panels
  static constexpr int NQA = SHARED ? 1 : (kAll + J - 1) / J;       // any panel
  static constexpr int SAN = SHARED ? kNear : NQN * J;              // X slabs held (the last ones zero), near
  static constexpr int SAA = SHARED ? kAll : NQA * J;               // any
  // A K chunk (8 rows) of an operand holds its slabs' columns, 16 bytes each, slab after slab.
  static constexpr unsigned LAN = 16u * SAN * KXP, LBN = SHARED ? 0u : 16u * kNear * KYP;
  static constexpr unsigned LAA = 16u * SAA * KXP, LBA = SHARED ? 0u : 16u * kAll * KYP;
  static constexpr unsigned up1024(unsigned b) { return (b + 1023u) & ~1023u; }
  static constexpr size_t bytes(int p) {  // two digit buffers, two staging buffers, two exponents a column
    return up1024(2u * (LAN + LBN) * (p / 8)) + 2 * (size_t)up1024(8u * COLS * p) + 2 * sizeof(int) * COLS;
  }
  // rows per panel that fit the warps and shared memory
  static constexpr int rows() {
    int p = 16;
    while (NCG * (p + 16) / 16 <= kConvWarps && bytes(p + 16) <= kSmemCap) p += 16;
    return p;
  }
};
template <int KXP_, int KYP_, bool SHARED_>
struct Plan : Geo<KXP_, KYP_, SHARED_> {
  using B = Geo<KXP_, KYP_, SHARED_>;
  static constexpr int P = B::rows();
  static constexpr unsigned b_off = B::LAN * (P / 8), dig_bytes = (B::LAN + B::LBN) * (P / 8);
  static constexpr unsigned stage_off = B::up1024(2 * dig_bytes), copy_bytes = 8u * B::COLS * P, stage_bytes = B::up1024(copy_bytes);
  // A panel with all slabs is multiplied in NF steps of at most FK K steps (16 rows)
  static constexpr int FK = (int)(dig_bytes / (2 * (B::LAA + B::LBA))), NF = (P / 16 + FK - 1) / FK;
  static constexpr unsigned b_off_all = B::LAA * (2 * FK);
  static constexpr int pairs_near = group_pairs(B::J, kNear, B::NQN), pairs_all = group_pairs(B::J, kAll, B::NQA);
  static constexpr size_t smem = B::bytes(P) + 1024;
  static_assert(FK >= 1 && NF >= 2 && P * pairs_near <= kPairRows && 16 * FK * pairs_all <= kPairRows, "a step fits the accumulators");
  static_assert(2 * (size_t)dig_bytes >= (SHARED_ ? 2u : 1u) * (size_t)(kLanes + 1) * KYP_ * 16, "final sums fit the digit buffers");
  static_assert(dig_bytes % 16 == 0 && B::LAA / 16 < (1u << 14), "descriptor strides");
};

__device__ __forceinline__ void st_digits(unsigned addr, unsigned a, unsigned b, unsigned c, unsigned d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// The ten near slabs of eight values (pairs m = rows 2m, 2m + 1) whose lane
// words are z, slab s at dst + s * stride.
__device__ __forceinline__ void store_near(unsigned dst, unsigned stride, const unsigned (&z)[4][5],
                                           const Sign2 (&sg)[4], unsigned e1024) {
#pragma unroll
  for (int i = 0; i < 5; ++i) {  // digits 2i (high bytes) and 2i + 1 (low bytes)
    const Sign2 s0 = i ? sg[0] : top(sg[0]), s1 = i ? sg[1] : top(sg[1]);
    const Sign2 s2 = i ? sg[2] : top(sg[2]), s3 = i ? sg[3] : top(sg[3]);
    st_digits(dst + (unsigned)(2 * i) * stride, digit_hi(z[0][i], e1024, s0), digit_hi(z[1][i], e1024, s1),
              digit_hi(z[2][i], e1024, s2), digit_hi(z[3][i], e1024, s3));
    st_digits(dst + (unsigned)(2 * i + 1) * stride, digit_lo(z[0][i], e1024, sg[0]), digit_lo(z[1][i], e1024, sg[1]),
              digit_lo(z[2][i], e1024, sg[2]), digit_lo(z[3][i], e1024, sg[3]));
  }
}

// The fourteen slabs: lane words z of the first ten digits, `low` (null: zero) of the last four.
__device__ __forceinline__ void store_all(unsigned dst, unsigned stride, const unsigned (&z)[4][5], const Sign2 (&sg)[4],
                                          const unsigned* low, unsigned e1024) {
  store_near(dst, stride, z, sg, e1024);
#pragma unroll 1
  for (int i = 0; i < 2; ++i) {
    const unsigned at = dst + (unsigned)(kNear + 2 * i) * stride;
    if (low) {
      st_digits(at, digit_hi(low[i], e1024, sg[0]), digit_hi(low[2 + i], e1024, sg[1]), digit_hi(low[4 + i], e1024, sg[2]),
                digit_hi(low[6 + i], e1024, sg[3]));
      st_digits(at + stride, digit_lo(low[i], e1024, sg[0]), digit_lo(low[2 + i], e1024, sg[1]),
                digit_lo(low[4 + i], e1024, sg[2]), digit_lo(low[6 + i], e1024, sg[3]));
    } else {
      st_digits(at, 0u, 0u, 0u, 0u);
      st_digits(at + stride, 0u, 0u, 0u, 0u);
    }
  }
}

// Lane words of the eight values' near digits and their signs.
template <bool ZERO>
__device__ __forceinline__ void near_lanes(const double (&v)[8], int A, unsigned (&z)[4][5], Sign2 (&sg)[4]) {
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    unsigned a1, a2, a3, b1, b2, b3;
    const double a = v[2 * m], b = v[2 * m + 1];
    near_words<ZERO>(a, 25 - A, a1, a2, a3);
    near_words<ZERO>(b, 25 - A, b1, b2, b3);
    sg[m] = sign2(a, b);
    z[m][0] = __byte_perm(a3, b3, 0x5410);
    z[m][1] = __byte_perm(a2, b2, 0x7632);
    z[m][2] = __byte_perm(a2, b2, 0x5410);
    z[m][3] = __byte_perm(a1, b1, 0x7632);
    z[m][4] = __byte_perm(a1, b1, 0x5410);
  }
}

// The same for any values, with the lane words of the last four digits in low.
__device__ __forceinline__ void any_lanes(const double (&v)[8], int A, unsigned (&z)[4][5], Sign2 (&sg)[4], unsigned* low) {
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    unsigned a[4], b[4];
    any_words(v[2 * m], A, a);
    any_words(v[2 * m + 1], A, b);
    sg[m] = sign2(v[2 * m], v[2 * m + 1]);
    z[m][0] = __byte_perm(a[3], b[3], 0x5410);
    z[m][1] = __byte_perm(a[2], b[2], 0x7632);
    z[m][2] = __byte_perm(a[2], b[2], 0x5410);
    z[m][3] = __byte_perm(a[1], b[1], 0x7632);
    z[m][4] = __byte_perm(a[1], b[1], 0x5410);
    low[2 * m] = __byte_perm(a[0], b[0], 0x7632);
    low[2 * m + 1] = __byte_perm(a[0], b[0], 0x5410);
  }
}

__device__ __forceinline__ double2 ld_shared2(unsigned addr) {
  double2 d;
  asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(d.x), "=d"(d.y) : "r"(addr));
  return d;
}

// Accumulators -> running sums (256 columns on) for the column blocks q, q + 4,
// .. of this warp's lanes (the four warps of a lane quarter share them out);
// accumulators back to zero.
template <int KYP>
__device__ __forceinline__ void drain(unsigned ta, int q) {
#pragma unroll 1
  for (int c = q; c <= kDiag; c += 4) {
    unsigned a[KYP], s[KYP];
    const unsigned t = ta + (unsigned)(c * KYP);
    tmem_ldn<KYP>(t, a);
    tmem_ldn<KYP>(t + 256u, s);
    tmem_waitn<KYP>(a);
    tmem_waitn<KYP>(s);
#pragma unroll
    for (int y = 0; y < KYP; ++y) s[y] += (unsigned)__float2int_rn(__uint_as_float(a[y]));
    tmem_stn<KYP>(t + 256u, s);
    tmem_zeron<KYP>(t);
  }
  tmem_wait_st();
}

// Running sums of this thread's TMEM lane (NY columns of every column block,
// from address ts) -> the totals.
// With h = sum_d S_d 2^(8 (14 - d)) the value is h 2^(Ax + Ay - 2168), and the
// total takes floor(h 2^-drop), sh = 8 jl + drop.  jl: the lane's digit phase
// (column block c holds diagonal c + jl), so h = 2^(-8 jl) sum_c S_c 2^(8 (14 - c))
// over c <= 14 - jl:
// four sums of neighbouring blocks in 64 bits each, five words, one shift.
// (Horner's rule on 128-bit integers took 12,000 to 18,000 cycles, most of a
// product of few rows.)  Out of line: its registers would cost the panel loop.
// LAST: the accumulators (256 columns before) are added in, not drained first.
template <class G, bool LAST>
__device__ __noinline__ void fold(unsigned ts, int jl, int sh, i128* tot) {
  constexpr int KYP = G::KYP, NY = KYP / 4;
#pragma unroll 1
  for (int y = 0; y < NY; ++y) {  // (one column at a time: few registers)
    unsigned s[kDiag + 1];
#pragma unroll
    for (int c = 0; c <= kDiag; ++c) tmem_ld1(ts + (unsigned)(c * KYP + y), s[c]);
    if constexpr (LAST) {
      unsigned f[kDiag + 1];
#pragma unroll
      for (int c = 0; c <= kDiag; ++c) tmem_ld1(ts - 256u + (unsigned)(c * KYP + y), f[c]);
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
      for (int c = 0; c <= kDiag; ++c) {  // no use moves above the wait
        asm volatile("" : "+r"(s[c]), "+r"(f[c]));
        s[c] += (unsigned)__float2int_rn(__uint_as_float(f[c]));
      }
    } else {
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
      for (int c = 0; c <= kDiag; ++c) asm volatile("" : "+r"(s[c]));
    }
#pragma unroll
    for (int part = 0; part < (G::SHARED ? 2 : 1); ++part) {  // SHARED: U from blocks c < J, V from the others
      // S_c 2^24 + S_c+1 2^16 + S_c+2 2^8 + S_c+3, a block outside the part or past the last diagonal as zero
      auto quad = [&](int c0) {
        long long r = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int c = c0 + u;
          if (c < 0 || (G::SHARED && (c < G::J) != (part == 0))) continue;
          const int x = c <= kDiag - (G::J - 1) || c + jl <= kDiag ? (int)s[c] : 0;  // (jl < J)
          asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(r) : "r"(x), "r"(1 << (24 - 8 * u)));
        }
        return r;
      };
      unsigned w[7];
      long long t = quad(11);
      w[0] = (unsigned)t;
      t = (t >> 32) + quad(7);
      w[1] = (unsigned)t;
      t = (t >> 32) + quad(3);
      w[2] = (unsigned)t;
      t = (t >> 32) + quad(-1);
      w[3] = (unsigned)t;
      w[4] = (unsigned)(t >> 32);
      w[5] = w[6] = (unsigned)((int)w[4] >> 31);
      unsigned a[5], o[4];
#pragma unroll
      for (int i = 0; i < 5; ++i) a[i] = sh < 32 ? w[i] : sh < 64 ? w[i + 1] : w[i + 2 < 7 ? i + 2 : 6];
#pragma unroll
      for (int i = 0; i < 4; ++i) o[i] = __funnelshift_r(a[i], a[i + 1], (unsigned)sh);
      tot[part * NY + y] += (i128)from_words(o[3], o[2], o[1], o[0]);
    }
  }
}

// The 16-column tile of a symmetric product whose columns are parts of rows.
struct PackPlan : Plan<16, 16, true> {};

// ------------------------------------------------------------ kernel
// PackPlan: a symmetric product of kx <= 2^lg <= 8 columns.  The rows are
// 16 >> lg parts of part_rows (n = part_rows here), and column c of part g is
// column g 2^lg + c of the 16-column tile, so that every lane converts; the
// diagonal blocks of the tile's product are the parts' products, whose sum is
// written.
template <class G, typename T, bool TMA>
__global__ void __launch_bounds__(kThreads, 1)
    umma_gram_partial_kernel(int64_t n, int kx, const T* __restrict__ X, int64_t ldx, int ky,
                             const T* __restrict__ Y, int64_t ldy, int64_t rows_per_chunk,
                             const __grid_constant__ CUtensorMap tmx, const __grid_constant__ CUtensorMap tmy,
                             FxPart* __restrict__ parts, const int* gate, int lg, int64_t part_rows) {
  static_assert(sizeof(T) == 8 || !TMA, "FP32 operands are copied by the converter threads");
  if (gate && *gate == 0) return;
  constexpr int KXP = G::KXP, KYP = G::KYP, J = G::J, P = G::P;
  constexpr bool SHARED = G::SHARED, PACK = std::is_same_v<G, PackPlan>;
  // Y columns of one draining thread (four warps share a TMEM lane quarter)
  constexpr int NY = KYP / 4;
  constexpr int kParts = SHARED ? 2 : 1;  // totals per output of a lane: U (and V)
  const int y0 = blockIdx.x * KYP;        // first Y column of the tile

  extern __shared__ __align__(1024) unsigned char smem_raw[];
  // 1024-byte aligned base (the 128-byte swizzle of the TMA boxes is anchored there)
  unsigned char* dig = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);  // 2 digit buffers
  unsigned char* stage = dig + G::stage_off;             // 2 staging buffers
  int* Erun = reinterpret_cast<int*>(stage + 2 * (size_t)G::stage_bytes);  // running exponents (0: none yet)
  int* Enew = Erun + G::COLS;                                              // the same with the current panel
  __shared__ __align__(8) unsigned long long full_bar[2], stage_bar[2], ready_bar[2];
  __shared__ unsigned tmem_base;
  __shared__ int flag, bad;
  // spec[p & 1]: 2 p + 1 if panel p holds a value above its column's exponent, else 2 p if one other
  // than zero below the near window (the largest wins); written before the arrivals for panel p - 1's last step
  __shared__ int spec[2], any_at;
  __shared__ __align__(8) unsigned long long cta_bar;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  // ---- set-up: TMEM (accumulators in columns 0..255, running sums in 256..511), barriers
  if (warp == 0) tmem_alloc(smem_u32(&tmem_base), 512);
  if (tid == kIssuer) {  // (the thread that fetches, so that the first copies need no CTA barrier)
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&full_bar[b]), 1);
      mbar_init(smem_u32(&stage_bar[b]), 1);
      mbar_init(smem_u32(&ready_bar[b]), kConvWarps);
      spec[b] = -1;
    }
    any_at = -1;
    mbar_init(smem_u32(&cta_bar), kWarps);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    flag = 0;
    bad = 0;
  }

  const int64_t r0 = (int64_t)blockIdx.y * rows_per_chunk;
  const int64_t r1 = min(n, r0 + rows_per_chunk);
  const int npan = r0 < r1 ? (int)((r1 - r0 + P - 1) / P) : 0;
  const unsigned dig_s = smem_u32(dig);
  const unsigned fb0 = smem_u32(&full_bar[0]);

  // ---- this thread's item: eight consecutive rows of one column of every panel
  const int cg = warp % G::NCG, kc = (warp / G::NCG) * 2 + (lane >> 4);  // column group, K chunk
  const int slot = cg * 16 + (lane & 15);      // column held
  const bool isb = !SHARED && cg * 16 >= KXP;  // of the Y operand (uniform over the warp)
  const int lc = slot - (isb ? KXP : 0);
  const bool mine = warp < kConvWarps && kc < P / 8 && slot < G::COLS;  // the thread has an item
  const int cx = PACK ? lc & ((1 << lg) - 1) : lc;  // column of X
  const bool valid = mine && (isb ? y0 + lc < ky : cx < kx);
  const unsigned dst_near = dig_s + (isb ? G::b_off + (unsigned)kc * G::LBN : (unsigned)kc * G::LAN) + (unsigned)lc * 16u;
  const unsigned e1024 = exp1024x2();

  // ---- staging: panel p's values in staging buffer p & 1, P / 16 boxes of
  // 16 rows (128 bytes, 128-byte swizzle) of X's columns, then of Y's.  TMA:
  // the last warp copies a whole panel (rows past the matrix read as zero, the
  // rows of the next chunk are masked).  Else (a base not 16-byte aligned, an
  // odd leading dimension, FP32) every converter thread copies its own item
  // into its own place, element by element.
  constexpr unsigned xbox = KXP * 128u, ybox = KYP * 128u;
  const unsigned stage_s = smem_u32(stage), sb0 = smem_u32(&stage_bar[0]);
  const T* src = valid ? (isb ? Y + (size_t)(y0 + lc) * ldy : X + (size_t)cx * ldx + (PACK ? (lc >> lg) * part_rows : 0)) + r0 + 8 * kc : nullptr;
  const unsigned item = (isb ? (P / 16) * xbox : 0u) + (unsigned)(kc >> 1) * (isb ? ybox : xbox) + (unsigned)lc * 128u;
  // 16-byte unit u (rows 2u, 2u + 1) of the item
  auto unit = [&](int p, int u) {
    return (unsigned)(p & 1) * G::stage_bytes + item + (((unsigned)(4 * (kc & 1) + u) ^ (unsigned)(lc & 7)) << 4);
  };
  auto fetch = [&](int p) {
    if constexpr (TMA) {
      if (tid == kIssuer) {
        const unsigned bar = sb0 + 8u * (unsigned)(p & 1), dst = stage_s + (unsigned)(p & 1) * G::stage_bytes;
        const int xr = (int)(r0 + (int64_t)p * P);
        fence_proxy_async();
        mbar_arrive_expect_tx(bar, G::copy_bytes);
        for (int h = 0; h < P / 16; ++h) {
          if (PACK) tma_load_3d(dst + (unsigned)h * xbox, &tmx, xr + 16 * h, bar);
          else tma_load_2d(dst + (unsigned)h * xbox, &tmx, xr + 16 * h, 0, bar);
          if (!SHARED) tma_load_2d(dst + (P / 16) * xbox + (unsigned)h * ybox, &tmy, xr + 16 * h, y0, bar);
        }
      }
    } else {
      // a copy of no bytes (a row past the chunk: the place is zero-filled)
      // names the partials array as its source, an address that is always valid
      const T* z = reinterpret_cast<const T*>(parts);
      const int64_t pr = (int64_t)p * P, left = r1 - (r0 + pr + 8 * kc);
      if (valid) {
#pragma unroll
        for (int m = 0; m < 8; ++m) {
          const unsigned d = stage_s + unit(p, m >> 1) + (unsigned)(m & 1) * 8u;
          if constexpr (sizeof(T) == 8) cp_async8z(d, m < left ? src + pr + m : z, m < left ? 8u : 0u);
          else cp_async4z(d, m < left ? src + pr + m : z, m < left ? 4u : 0u);
        }
      }
      cp_async_commit_group();
    }
  };
  // Panel p's values (zeros past the chunk).  The units of an item differ in
  // bits 4 and 5 of their address only (the swizzle's), as an exclusive or.
  double v[8];
  // rows of this thread's item that panel p has (8 or more but in the chunk's last panel)
  auto rows_left = [&](int p) { return (int)min(r1 - (r0 + (int64_t)p * P + 8 * kc), (int64_t)8); };
  const unsigned item_s = stage_s + (mine ? unit(0, 0) : 0u);
  auto load = [&](int p) {
    if constexpr (TMA) mbar_wait(sb0 + 8u * (unsigned)(p & 1), (unsigned)(p >> 1) & 1u, &bad);
    else asm volatile("cp.async.wait_group 1;" ::: "memory");  // p + 1's may be in flight
    const unsigned at = item_s + (unsigned)(p & 1) * G::stage_bytes;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const double2 d = ld_shared2(at ^ ((unsigned)m << 4));
      if constexpr (sizeof(T) == 8) {
        v[2 * m] = d.x;
        v[2 * m + 1] = d.y;
      } else {
        v[2 * m] = widen(__int_as_float(__double2loint(d.x)));
        v[2 * m + 1] = widen(__int_as_float(__double2loint(d.y)));
      }
    }
    if (TMA && p + 1 == npan) {  // (the copies zero-fill rows past the chunk, but not the tensor map)
      const int left = rows_left(p);
#pragma unroll
      for (int m = 0; m < 8; ++m)
        if (m >= left) v[m] = 0.0;
    }
  };
  // The column's window: a value is near when (2 |hi word| - wlo) < wrange, unsigned.
  int te = 0;  // running exponent of this thread's column (0: none)
  unsigned wlo = 0, wrange = valid ? 0u : 0xffffffffu;
  auto set_window = [&]() {
    const int A = max(te, 1), f = max(A - kNearBits, 1);
    wlo = (unsigned)f << 21;
    wrange = ((unsigned)(A + 1) << 21) - wlo;
  };
  // Whether a value lies above it.  Over the warp: `zeros`, a value that is zero
  // (rows past the chunk's end in its last panel among them) or below it, `below`,
  // one other than zero below it; the warp cuts its values accordingly.
  bool zeros = false, below = false;
  auto look = [&]() {
    unsigned k = 0;
#pragma unroll
    for (int m = 0; m < 8; ++m) k = max(k, 2u * hi32(v[m]) - wlo);
    zeros = __any_sync(0xffffffffu, k >= wrange);
    below = false;
    if (!zeros) return false;
    bool up = false, low = false;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const unsigned a = hi32(v[m]) & 0x7fffffffu;
      const bool out = 2u * hi32(v[m]) - wlo >= wrange && (a | lo32(v[m])) != 0u;
      const bool above = 2u * a >= wlo;
      up |= out && above;
      low |= out && !above;
    }
    below = __any_sync(0xffffffffu, low);
    return up;
  };
  // the values of a panel that `below` holds for, the lane words of their digits
  // 10..13, and the barriers passed in the panel loop; touched rarely, so they are
  // kept out of registers
  struct {
    double v[8];
    unsigned low[8], syncs;
  } rare_, *rare = &rare_;
  asm volatile("" : "+l"(rare)::"memory");
  rare->syncs = 0;
  if (npan > 0) {
    fetch(0);
    if (!TMA || npan > 1) fetch(1);
  }

  // zero digits (padded columns and slabs stay zero) and exponents, while the first copies fly
  for (int c = tid; c < 2 * G::COLS; c += kThreads) Erun[c] = 0;  // Erun and Enew
  if (kx < (PACK ? 1 << lg : KXP) || (!SHARED && ky - y0 < KYP)) {
    for (unsigned e = tid; e < 2 * G::dig_bytes / 16; e += kThreads)
      reinterpret_cast<uint4*>(dig)[e] = make_uint4(0u, 0u, 0u, 0u);
  } else if constexpr (G::SAN > kNear) {  // the slabs past the last digit of every K chunk (the others are stored)
    constexpr unsigned per = (G::SAN - kNear) * KXP;
    for (unsigned e = tid; e < 2 * (P / 8) * per; e += kThreads) {
      const unsigned c = e / per, u = e % per;  // chunk of the two buffers
      reinterpret_cast<uint4*>(dig + (c / (P / 8)) * G::dig_bytes + (c % (P / 8)) * G::LAN)[kNear * KXP + u] =
          make_uint4(0u, 0u, 0u, 0u);
    }
  }
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const unsigned taddr = tmem_base;

  // ---- drains: this thread's TMEM lane: lane block jl (digit phase), X column xl
  const int Lq = (warp & 3) * 32, L = Lq + lane;
  const int jl = L / KXP, xl = L % KXP;
  const int yq = (warp >> 2) * NY;  // first of this thread's NY Y columns
  const unsigned tq = taddr + ((unsigned)Lq << 16);             // the lane quarter's columns
  const unsigned tsum = tq + (unsigned)yq + 256u;               // the running sums of its columns
  // the exact totals; touched once per fold, so they are kept out of registers
  i128 totals[kParts * NY];
  i128* tot = totals;
  asm volatile("" : "+l"(tot)::"memory");
  for (int y = 0; y < kParts * NY; ++y) tot[y] = 0;
  // bits of h that a total drops: 127 hold the sum of the chunk's rows (PACK: of all parts)
  auto drop = [&]() { return fold_bits((unsigned)rows_per_chunk * (PACK ? 16u >> lg : 1u)); };

  // the running sums and, first, the accumulators at zero (this warp's share of the column blocks)
  auto zero_blocks = [&](unsigned t) {
#pragma unroll 1
    for (int c = warp >> 2; c <= kDiag; c += 4) tmem_zeron<KYP>(t + (unsigned)(c * KYP));
    tmem_wait_st();
  };
  zero_blocks(tq);
  zero_blocks(tq + 256u);
  tc_fence_before();

  // ---- steps: one digit buffer filled and multiplied (a near panel, or half
  // of a panel with all slabs).  Step `step` uses buffer step & 1.
  int step = 0;          // steps converted so far
  int pend = 0;          // K steps (16 rows) of the last converted step, not issued yet (0: none)
  bool pend_all = false; // ... with all slabs
  int used = 0;          // row-pairs (of kPairRows) the accumulators hold, the pending step included
  int drains = 0;        // since the last fold
  auto issue = [&]() {   // the pending step's MMAs (after a barrier that follows its stores)
    if (pend > 0 && tid == kIssuer) {
      tc_fence_after();
      const int b = (step - 1) & 1;
      const unsigned ab = dig_s + (unsigned)b * G::dig_bytes;
      if (!pend_all) {
        for (int ks = 0; ks < pend; ++ks) {
          const unsigned long long bd = SHARED ? sdesc(ab + (unsigned)ks * 2u * G::LAN, G::LAN, 128u)
                                               : sdesc(ab + G::b_off + (unsigned)ks * 2u * G::LBN, G::LBN, 128u);
#pragma unroll
          for (int q = 0; q < G::NQN; ++q) {
            constexpr int even = KYP == 8 ? 1 : 0;  // N is a multiple of 16
            const int nt = (min(kNear, kDiag + 1 - J * q) + even) & ~even;
            mma_f16(taddr + (unsigned)(KYP * J * q),
                    sdesc(ab + (unsigned)(J * q * KXP) * 16u + (unsigned)ks * 2u * G::LAN, G::LAN, 128u), bd,
                    idesc_f16(kLanes, KYP * nt), 1u);  // the accumulators start at zero and drains zero them
          }
        }
      } else {
        for (int ks = 0; ks < pend; ++ks) {
          const unsigned long long bd = SHARED ? sdesc(ab + (unsigned)ks * 2u * G::LAA, G::LAA, 128u)
                                               : sdesc(ab + G::b_off_all + (unsigned)ks * 2u * G::LBA, G::LBA, 128u);
#pragma unroll 1
          for (int q = 0; q < G::NQA; ++q) {
            constexpr int even = KYP == 8 ? 1 : 0;
            const int nt = (min(kAll, kDiag + 1 - J * q) + even) & ~even;
            mma_f16(taddr + (unsigned)(KYP * J * q),
                    sdesc(ab + (unsigned)(J * q * KXP) * 16u + (unsigned)ks * 2u * G::LAA, G::LAA, 128u), bd,
                    idesc_f16(kLanes, KYP * nt), 1u);
          }
        }
      }
      mma_commit(fb0 + 8u * b);
    }
    pend = 0;
  };
  // wait for the MMAs of step s (committed to its buffer's barrier)
  // Barrier of the panel loop over all warps, bounded like every wait in it, so
  // that warps which a wait that ran out has sent out of the loop hold up nobody.
  auto sync_all = [&]() {
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&cta_bar));
    mbar_wait(smem_u32(&cta_bar), rare->syncs++ & 1u, &bad);
  };
  auto wait_step = [&](int s) { mbar_wait(fb0 + 8u * (unsigned)(s & 1), (unsigned)(s >> 1) & 1u, &bad); };
  // Empties the accumulators (after the MMAs of the steps before s) and, when
  // due or asked for, folds the running sums.
  auto empty = [&](int s, bool full) {
    ++drains;
    full |= drains >= kFoldDrains;
    wait_step(s - 1);
    tc_fence_after();
    drain<KYP>(tq, warp >> 2);
    if (full) {  // all of the lane quarter's blocks are drained
      tc_fence_before();
      sync_all();
      tc_fence_after();
      fold<G, false>(tsum, jl, 8 * jl + drop(), tot);
      tc_fence_before();
      sync_all();
      tc_fence_after();
      zero_blocks(tq + 256u);
    }
    tc_fence_before();
    if (full) drains = 0;
    used = 0;
  };
  // the step just converted (cost row-pairs) becomes the pending one; the
  // accumulators are emptied first when they could not hold it
  auto finish_step = [&](int ks, bool all, int cost) {
    fence_proxy_async();
    if (used + cost > kPairRows) empty(step, false);
    used += cost;
    pend = ks;
    pend_all = all;
    ++step;
  };

  int dirty = 0;  // bit b: buffer b was last used with all slabs (its zero slabs and columns are to be zeroed again)

  // the near digits of this thread's item into step `step`'s buffer
  auto put = [&](const unsigned (&z)[4][5], const Sign2 (&sg)[4]) {
    const unsigned at = dst_near + (unsigned)(step & 1) * G::dig_bytes;
    if (mine) {
      if (step >= 2) wait_step(step - 2);  // the buffer's last MMAs are done
      if (valid) {
        if (isb) store_near(at, 16u * KYP, z, sg, e1024);
        else store_near(at, 16u * KXP, z, sg, e1024);
      }
      if ((dirty >> (step & 1)) & 1) {  // zero slabs, and the padded columns
        const unsigned st = 16u * (unsigned)(isb ? KYP : KXP);
        const int s1 = isb || SHARED ? kNear : G::SAN;
        for (int s = valid ? kNear : 0; s < s1; ++s) st_digits(at + (unsigned)s * st, 0u, 0u, 0u, 0u);
      }
    }
    dirty &= ~(1 << (step & 1));
  };
  // One panel: convert panel p (its values are in v), take panel p + 1's values
  // and look whether they are near, then, once every warp has stored the step
  // before (ready), store the digits and arrive.  The last warp issues that
  // step's MMAs and the copies of panel p + 1's successor at that point instead.
  const bool conv = warp < kConvWarps;
  const unsigned rb0 = smem_u32(&ready_bar[0]);
  auto wait_ready = [&](int s) { return mbar_wait(rb0 + 8u * (unsigned)(s & 1), (unsigned)(s >> 1) & 1u, &bad); };
  auto arrive = [&]() {  // this warp's digits of the last step are stored
    __syncwarp();
    if (conv && lane == 0) mbar_arrive(rb0 + 8u * (unsigned)((step - 1) & 1));
  };
  if (npan > 0) {  // the columns' exponents from panel 0
    if (conv) {
      load(0);
      unsigned m = 0;  // largest magnitude
#pragma unroll
      for (int i = 0; i < 8; ++i) m = max(m, abs_hi(v[i]));
      const int e = (int)(m >> 20);  // (subnormals set none: an alignment exponent is at least 1)
      if (valid && e > 0) {
        if (e == 2047) flag = 1;
        // (finite exponents stay below 2047, so that an Inf or NaN always raises)
        atomicMax(&Enew[slot], e == 2047 ? e : min(e + EO_GRAM_HEADROOM, 2046));
      }
    }
    __syncthreads();
    if (tid < G::COLS) Erun[tid] = Enew[tid];
    if (valid) {
      te = Enew[slot];
      set_window();
    }
    if (conv) {
      look();  // (nothing above: the exponents are the panel's)
      if (below && lane == 0) atomicMax(&spec[0], 0);
    }
  }
  __syncthreads();
  if (TMA && npan > 2) fetch(2);  // (TMA: panel 0's values are in registers)
  int p = 0;
#pragma unroll 1
  for (; p < npan; ++p) {
    unsigned z[4][5];
    Sign2 sg[4];
    bool up = false, cut_all = below;
    if (conv) {
      if (below) {  // cut below, where every warp is known to take that branch
#pragma unroll
        for (int i = 0; i < 8; ++i) rare->v[i] = v[i];
      }
      if (zeros) near_lanes<true>(v, max(te, 1), z, sg);
      else near_lanes<false>(v, max(te, 1), z, sg);
      if constexpr (!TMA) fetch(p + 2);
      if (p + 1 < npan) {
        load(p + 1);
        up = look();
      }
    }
    if (step > 0) {
      // (a wait that ran out: the whole warp leaves; nothing in the loop waits for it without a bound)
      if (!__all_sync(0xffffffffu, wait_ready(step - 1))) break;
      if (!conv) {
        // every warp has taken panel p's values: its staging buffer is free
        if (TMA && p + 2 < npan) fetch(p + 2);
        issue();  // the last step's
      }
    }
    int ks = P / 16, cost = P * G::pairs_near;
    bool all = false;
    // (Nobody writes this word for panel p + 2 before the last warp has read it:
    // a converter that has something to write waits for MMAs first that the last
    // warp issues after this, or stands in panel p's barriers.)
    const int sp = *reinterpret_cast<volatile int*>(&spec[p & 1]);
    if ((sp >> 1) == p) {
      // Panel p is not near: every warp comes here.
      const bool grow = sp & 1;
      if (grow) {
        sync_all();
        double u[8];
        unsigned m = 0;  // largest magnitude
        const int64_t pr = (int64_t)p * P;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          u[i] = (valid && r0 + pr + 8 * kc + i < r1) ? (sizeof(T) == 8 ? (double)src[pr + i] : widen((float)src[pr + i])) : 0.0;
          m = max(m, abs_hi(u[i]));
        }
        // exponents (subnormals never raise a column: its alignment exponent is at least 1)
        if (valid && m >= ((unsigned)te + 1u) << 20) {
          const int e = (int)(m >> 20);
          if (e == 2047) flag = 1;
          // (finite exponents stay below 2047, so that an Inf or NaN always raises)
          atomicMax(&Enew[slot], e == 2047 ? e : min(e + EO_GRAM_HEADROOM, 2046));
        }
        sync_all();
        if (used > 0) {
          empty(step, true);
          // totals onto the new grid: divide by 2^(growth of both columns' exponents)
          const int ysb = SHARED ? 0 : KXP;
          for (int y = 0; y < NY; ++y) {
            const int cy = ysb + yq + y;
            // (a column of zeros and subnormals so far, exponent 0, stands on the grid of exponent 1)
            const int dx = max(Enew[xl], 1) - max(Erun[xl], 1);
            const int dy = max(Enew[cy], 1) - max(Erun[cy], 1);
            for (int q = 0; q < kParts; ++q) tot[q * NY + y] = w_shift(tot[q * NY + y], dx + dy);
          }
        }
        sync_all();
        if (tid < G::COLS) Erun[tid] = Enew[tid];
        if (valid) {
          te = Enew[slot];
          set_window();
        }
        // a nonzero value (normal or not) below the window
        const unsigned floor = near_floor(max(te, 1));
        cut_all = false;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          cut_all |= valid && (abs_hi(u[i]) | lo32(u[i])) != 0u && abs_hi(u[i]) < floor;
          rare->v[i] = u[i];
        }
        cut_all = __any_sync(0xffffffffu, cut_all);
        if (cut_all && lane == 0) *reinterpret_cast<volatile int*>(&any_at) = p;
        sync_all();
        all = *reinterpret_cast<volatile int*>(&any_at) == p;
        near_lanes<true>(u, max(te, 1), z, sg);
      } else {
        all = true;
      }
      if (!all) {
        put(z, sg);
      } else {
        // All digits: the panel in NF steps, the items of a step's K chunks each.
        if (cut_all) {
          double u[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) u[i] = rare->v[i];
          any_lanes(u, max(te, 1), z, sg, rare->low);
        }
#pragma unroll 1
        for (int h = 0; h < G::NF; ++h) {
          if (h) {  // the step before is stored: its MMAs
            finish_step(G::FK, true, 16 * G::FK * G::pairs_all);
            arrive();
            wait_ready(step - 1);
            issue();
          }
          const int k = kc - h * 2 * G::FK;  // K chunk within the step
          if (mine && k >= 0 && k < 2 * G::FK) {
            if (step >= 2) wait_step(step - 2);
            const unsigned dst = dig_s + (unsigned)(step & 1) * G::dig_bytes +
                                 (isb ? G::b_off_all + (unsigned)k * G::LBA : (unsigned)k * G::LAA) + (unsigned)lc * 16u;
            const unsigned st = 16u * (unsigned)(isb ? KYP : KXP);
            if (valid) store_all(dst, st, z, sg, cut_all ? rare->low : nullptr, e1024);
            for (int s = valid ? kAll : 0; s < (isb ? kAll : G::SAA); ++s) st_digits(dst + (unsigned)s * st, 0u, 0u, 0u, 0u);
          }
          dirty |= 1 << (step & 1);
        }
        ks = P / 16 - (G::NF - 1) * G::FK;
        cost = 16 * ks * G::pairs_all;
      }
      // panel p + 1's values again (they are still staged; nothing but the
      // loop's state is kept across this branch) and their look, as the
      // exponents may have grown
      if (conv && p + 1 < npan) {
        load(p + 1);
        up = look();
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = 0.0;
      }
    } else {
      put(z, sg);
    }
    finish_step(ks, all, cost);
    if (conv && (up || below)) {
      if (up) atomicMax(&spec[(p + 1) & 1], 2 * p + 3);
      else if (lane == 0) atomicMax(&spec[(p + 1) & 1], 2 * p + 2);
    }
    arrive();
  }

  if constexpr (!TMA) asm volatile("cp.async.wait_all;" ::: "memory");  // the last (empty) copies
  // the last step's MMAs, drain and fold
  __syncthreads();
  issue();
  if (tid == kIssuer && *reinterpret_cast<volatile int*>(&bad)) {
    // after a wait that ran out: this thread's own MMAs and copies end before TMEM and shared memory are released
    if (step > 0) mbar_wait_final(fb0 + 8u * (unsigned)((step - 1) & 1), (unsigned)((step - 1) >> 1) & 1u, &bad);
    // (at panel p the copies before panel p + 2 are issued, one phase of each buffer's barrier unwaited at most)
    for (int f = min(p + 2, npan), q = max(f - 2, 0); TMA && q < f; ++q) mbar_wait_final(sb0 + 8u * (unsigned)(q & 1), (unsigned)(q >> 1) & 1u, &bad);
  }
  if (step > 0) {
    if (warp == 0) mbar_wait_final(fb0 + 8u * (unsigned)((step - 1) & 1), (unsigned)((step - 1) >> 1) & 1u, &bad);
    wait_step(step - 1);
    tc_fence_after();  // (the drains' running sums: before the barrier above)
    fold<G, true>(tsum, jl, 8 * jl + drop(), tot);
    tc_fence_before();
  }
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(taddr, 512);
  }

  // sum the lane blocks (digit phase j) of every output and write the partials
  // (lanes next to one another, and a lane of padding: neither the stores nor
  // the loads of a column or of its transpose meet in a bank)
  constexpr int kRow = kLanes + 1;
  i128* red = reinterpret_cast<i128*>(dig);  // kParts x KYP x 129 entries (the MMAs are done)
  for (int q = 0; q < kParts; ++q)
    for (int y = 0; y < NY; ++y) red[(q * KYP + yq + y) * kRow + L] = tot[q * NY + y];
  __syncthreads();
  auto output = [&](int i, int yo) {  // columns i and yo of the tile
    i128 w = 0;
    for (int b = 0; b < J; ++b) {
      w += red[yo * kRow + b * KXP + i];
      if constexpr (SHARED) w += red[(KYP + yo) * kRow + b * KXP + i] + red[(KYP + i) * kRow + b * KXP + yo];
    }
    FxPart o;
    o.wl = (long long)(unsigned long long)(u128)w;
    o.wh = (long long)(w >> 64);
    o.s = max(Erun[i], 1) + max(Erun[(SHARED ? 0 : KXP) + yo], 1) - kOffsetDigits + drop();
    o.flag = flag | bad;
    o.pad = 0;
    return o;
  };
  FxPart* mine_parts = parts + (size_t)blockIdx.y * ((size_t)kx * ky);
  if constexpr (PACK) {  // the parts' blocks, aligned to the largest scale
    FxPart* blocks = reinterpret_cast<FxPart*>(stage);  // (the copies are done)
    const int kc2 = 1 << lg;
    for (int e = tid; e < 16 << lg; e += kThreads) {
      const int i = e & 15, yo = (i & -kc2) + (e >> 4);
      blocks[e] = output(i, yo);
    }
    __syncthreads();
    for (int e = tid; e < kx * kx; e += kThreads) {
      const int i = e % kx, j = e / kx;
      FxPart o = blocks[j * 16 + i];
      for (int g = kc2; g < 16; g += kc2) o.s = max(o.s, blocks[j * 16 + g + i].s);
      i128 w = 0;
      for (int g = 0; g < 16; g += kc2) {
        const FxPart& b = blocks[j * 16 + g + i];
        w += w_shift((i128)(((u128)(unsigned long long)b.wh << 64) | (unsigned long long)b.wl), o.s - b.s);
      }
      o.wl = (long long)(unsigned long long)(u128)w;
      o.wh = (long long)(w >> 64);
      mine_parts[j * kx + i] = o;
    }
  } else {
    for (int e = tid; e < KXP * KYP; e += kThreads) {
      const int i = e % KXP, yo = e / KXP, j = y0 + yo;
      if (i < kx && j < ky) mine_parts[(size_t)j * kx + i] = output(i, yo);
    }
  }
}

// ------------------------------------------------------------ host side
// Tile and launch geometry of one product: X tile width kxp >= kx (16, 32 or
// 64), Y tile width kyp, row chunks.
struct UPlan {
  int kxp, kyp, nty;
  bool shared;
};

UPlan make_plan(int kx, int ky, bool sym) {
  UPlan p{};
  p.shared = sym && kx <= 16;
  p.kxp = kx <= 16 ? 16 : (kx <= 32 ? 32 : 64);
  p.kyp = p.shared || ky > 8 ? 16 : 8;
  p.nty = p.shared ? 1 : (ky + p.kyp - 1) / p.kyp;
  return p;
}

constexpr int kMinRows = 64;  // rows of the smallest row chunk

// A symmetric product with more than 16 columns runs as column strips of 16
// (below), from kStripRows rows on; with fewer, as one launch of X^T X: it
// converts more, but the strips run one after another, each with its fixed part
// (set-up, first panel, last fold: 10 us and the reduction's 5 to 9).
// Measured, one launch vs strips: 2e4 rows of 32 columns 32 vs 57 us, of 64 49
// vs 114; 1e5 rows 61 vs 81, 131 vs 161; 2e5 rows 101 vs 98, 234 vs 253.
constexpr int64_t kStripRows = 160000;
bool use_strips(int64_t n, int kx, bool sym) { return sym && kx > 16 && n >= kStripRows; }

int num_chunks(int64_t n, const UPlan& p) {
  const int64_t by_rows = (n + kMinRows - 1) / kMinRows;
  // one CTA per SM, none left over for a second wave (three tiles with 51
  // chunks: a symmetric product of 48 columns on 1e5 rows took 156 us, on 64 131)
  const int64_t want = std::max<int64_t>(1, 152 / p.nty);
  const int64_t need = (n + (1ll << 22) - 1) >> 22;                       // <= 2^22 rows per chunk
  return (int)std::max<int64_t>(1, std::min(by_rows, std::max(want, need)));
}

// Row chunks under a cap of ctas CTAs (0 = none): never more than num_chunks
// (the scratch is sized for it), never fewer than the 2^22-row bound needs.
int capped_chunks(int64_t n, const UPlan& p, int ctas) {
  const int c = num_chunks(n, p);
  if (ctas <= 0) return c;
  const int64_t need = (n + (1ll << 22) - 1) >> 22;
  const int64_t cap = std::max<int64_t>(1, ctas / p.nty);
  return (int)std::max<int64_t>(std::max<int64_t>(1, need), std::min<int64_t>(c, cap));
}

PFN_cuTensorMapEncodeTiled_v12000 encode_tiled() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
  });
  return fn;
}

// Tensor map of a column-major n-by-k FP64 matrix: boxes of 16 rows x w columns.
bool make_map(CUtensorMap* m, const double* A, int64_t n, int k, int64_t ld, int w) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = encode_tiled();
  if (!enc) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)std::max<int64_t>(n, 1), (cuuint64_t)k};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * 8u};
  const cuuint32_t box[2] = {16u, (cuuint32_t)w};
  const cuuint32_t estr[2] = {1u, 1u};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 2, const_cast<double*>(A), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The same for a matrix in parts of q rows, one above the other: boxes of 16
// rows x kc columns x all parts.
bool make_parts_map(CUtensorMap* m, const double* A, int64_t q, int k, int64_t ld, int kc, int parts) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = encode_tiled();
  if (!enc) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)q, (cuuint64_t)k, (cuuint64_t)parts};
  const cuuint64_t strides[2] = {(cuuint64_t)ld * 8u, (cuuint64_t)q * 8u};
  const cuuint32_t box[3] = {16u, (cuuint32_t)kc, (cuuint32_t)parts};
  const cuuint32_t estr[3] = {1u, 1u, 1u};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 3, const_cast<double*>(A), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct Maps {
  CUtensorMap x, y;
};

template <class G, typename T, bool TMA>
cudaError_t launch_kernel(const UPlan& plan, int chunks, int64_t n, int kx, const T* X, int64_t ldx, int ky,
                          const T* Y, int64_t ldy, int64_t rpc, const Maps& maps, FxPart* parts, const int* gate,
                          cudaStream_t st, int lg = 0, int64_t part_rows = 0) {
  cudaError_t e = set_dyn_smem(umma_gram_partial_kernel<G, T, TMA>, G::smem);
  if (e != cudaSuccess) return e;
  umma_gram_partial_kernel<G, T, TMA>
      <<<dim3(plan.nty, chunks), kThreads, G::smem, st>>>(n, kx, X, ldx, ky, Y, ldy, rpc, maps.x, maps.y, parts, gate,
                                                       lg, part_rows);
  return cudaGetLastError();
}

template <typename T, bool TMA>
cudaError_t launch_plan(const UPlan& plan, int chunks, int64_t n, int kx, const T* X, int64_t ldx, int ky,
                        const T* Y, int64_t ldy, int64_t rpc, const Maps& maps, FxPart* parts, const int* gate,
                        cudaStream_t st) {
#define EO_UMMA_LAUNCH(A, B, S) \
  return launch_kernel<Plan<A, B, S>, T, TMA>(plan, chunks, n, kx, X, ldx, ky, Y, ldy, rpc, maps, parts, gate, st)
  if (plan.shared) EO_UMMA_LAUNCH(16, 16, true);
  if (plan.kyp == 16) {
    if (plan.kxp == 16) EO_UMMA_LAUNCH(16, 16, false);
    if (plan.kxp == 32) EO_UMMA_LAUNCH(32, 16, false);
    EO_UMMA_LAUNCH(64, 16, false);
  }
  if (plan.kxp == 16) EO_UMMA_LAUNCH(16, 8, false);
  if (plan.kxp == 32) EO_UMMA_LAUNCH(32, 8, false);
  EO_UMMA_LAUNCH(64, 8, false);
#undef EO_UMMA_LAUNCH
}

// One thread waits for a phase of an mbarrier that nothing completes, bounded
// by limit_ns: the bounded-wait path of the tensor-core kernels, exercised on
// its own (it records the expiry like any other wait that runs out).
__global__ void wait_selftest_kernel(unsigned long long limit_ns) {
  __shared__ __align__(8) unsigned long long bar;
  __shared__ int abort_flag;
  if (threadIdx.x != 0) return;
  abort_flag = 0;
  mbar_init(smem_u32(&bar), 1);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  (void)mbar_wait(smem_u32(&bar), 0u, &abort_flag, limit_ns);
}

}  // namespace

cudaError_t umma_wait_selftest(unsigned long long limit_ns, cudaStream_t st) {
  wait_selftest_kernel<<<1, 32, 0, st>>>(limit_ns);
  return cudaGetLastError();
}

cudaError_t umma_gram_take_wait_record(unsigned* out) { return take_wait_record(out); }

namespace {

// A symmetric product with more than 16 columns runs as column strips of 16:
// strip c0 .. c1 - 1 is X[:, 0:c1]^T X[:, c0:c1] (the first one the symmetric
// 16-column product), of which the reduction keeps the entries on and above
// the diagonal of G and mirrors them (so G is exactly symmetric).  Each
// value is converted once per strip that reads it, where one-tile plans of
// X^T Y over all columns convert it once per 16-column Y tile and once more
// as the Y operand.
template <typename T>
cudaError_t launch_one(int64_t n, int kx, const T* X, int64_t ldx, int ky, const T* Y, int64_t ldy, void* scratch,
                       double* G_hi, double* G_lo, int ldg, const int* gate, cudaStream_t st, int ctas, bool sym,
                       int jo, bool shared) {
  const UPlan plan = make_plan(kx, ky, shared);
  const int chunks = capped_chunks(n, plan, ctas);
  // whole K steps per chunk: at most 15 rows of imbalance, and every chunk's
  // first row keeps its column's alignment
  int64_t rpc = (n + chunks - 1) / chunks;
  rpc = std::max<int64_t>(16, (rpc + 15) / 16 * 16);
  FxPart* parts = static_cast<FxPart*>(scratch);
  alignas(64) Maps maps{};
  cudaError_t e;
  bool tma = false;
  if constexpr (sizeof(T) == 8) {
    // TMA addresses 16-byte aligned bases and leading dimensions of whole
    // 16-byte units, rows below 2^31 (a box may start past the last row)
    const char* lm = getenv("EO_DD_GRAM_LOADS");  // "direct": the threads' own copies for such operands too
    tma = (uintptr_t)X % 16 == 0 && (uintptr_t)Y % 16 == 0 && ldx % 2 == 0 && ldy % 2 == 0 && n < (1ll << 31) - 1024 &&
          !(lm && lm[0] == 'd') && make_map(&maps.x, X, n, kx, ldx, plan.kxp) &&
          make_map(&maps.y, Y, n, ky, ldy, plan.kyp);
    e = tma ? launch_plan<T, true>(plan, chunks, n, kx, X, ldx, ky, Y, ldy, rpc, maps, parts, gate, st)
            : launch_plan<T, false>(plan, chunks, n, kx, X, ldx, ky, Y, ldy, rpc, maps, parts, gate, st);
  } else {
    e = launch_plan<T, false>(plan, chunks, n, kx, X, ldx, ky, Y, ldy, rpc, maps, parts, gate, st);
  }
  if (e != cudaSuccess) return e;
  return launch_fx_reduce(kx, ky, sym, chunks, parts, G_hi, G_lo, ldg, gate, st, jo);
}

// Symmetric products of up to 8 columns: the rows in 16 >> lg parts side by side
// as the columns of the 16-column tile, so that its lanes all have a value; the
// fewer than 16 rows a part that are left over go through the integer limbs, a
// launch of 8 us that pays from kPackRows rows on.  Measured: 32e6 rows of 4
// columns 1.43 ms (limbs; 2.1 on a padded tile) -> 0.49; 4e6 rows of 8 columns
// 282 us (padded tile) -> 145.
int pack_lg(int kx) { return kx <= 1 ? 0 : (kx <= 2 ? 1 : (kx <= 4 ? 2 : 3)); }
constexpr int64_t kPackRows = 300000;
int64_t part_rows_of(int64_t n, int kx);
bool use_pack(int64_t n, int kx, bool sym) {
  return sym && kx <= 8 && n >= 256 && (n >= kPackRows || n == (16 >> pack_lg(kx)) * part_rows_of(n, kx));
}
int64_t part_rows_of(int64_t n, int kx) { return n / (16 * (16 >> pack_lg(kx))) * 16; }

cudaError_t launch_packed(int64_t n, int kx, const double* X, int64_t ldx, void* scratch, double* G_hi, double* G_lo,
                          int ldg, const int* gate, cudaStream_t st, int ctas) {
  const int lg = pack_lg(kx), np = 16 >> lg;
  const int64_t q = part_rows_of(n, kx), rest = n - np * q;
  const UPlan plan = make_plan(kx, kx, true);
  const int chunks = capped_chunks(q, plan, ctas);
  int64_t rpc = (q + chunks - 1) / chunks;
  rpc = std::max<int64_t>(16, (rpc + 15) / 16 * 16);
  FxPart* parts = static_cast<FxPart*>(scratch);
  alignas(64) Maps maps{};
  using P = PackPlan;
  const char* lm = getenv("EO_DD_GRAM_LOADS");
  const bool tma = (uintptr_t)X % 16 == 0 && ldx % 2 == 0 && n < (1ll << 31) - 1024 && !(lm && lm[0] == 'd') &&
                   make_parts_map(&maps.x, X, q, kx, ldx, 1 << lg, np);
  cudaError_t e =
      tma ? launch_kernel<P, double, true>(plan, chunks, q, kx, X, ldx, kx, X, ldx, rpc, maps, parts, gate, st, lg, q)
          : launch_kernel<P, double, false>(plan, chunks, q, kx, X, ldx, kx, X, ldx, rpc, maps, parts, gate, st, lg, q);
  if (e != cudaSuccess) return e;
  if (rest > 0) {
    e = launch_fx_gram_part(rest, kx, X + np * q, ldx, parts + (size_t)chunks * kx * kx, gate, st);
    if (e != cudaSuccess) return e;
  }
  return launch_fx_reduce(kx, kx, true, chunks + (rest > 0 ? 1 : 0), parts, G_hi, G_lo, ldg, gate, st, 0);
}

template <typename T>
cudaError_t launch_gram_t(int64_t n, int kx, const T* X, int64_t ldx, int ky, const T* Y, int64_t ldy, bool sym,
                          void* scratch, double* G_hi, double* G_lo, int ldg, const int* gate, cudaStream_t st,
                          int ctas) {
  if constexpr (sizeof(T) == 8) {
    if (use_pack(n, kx, sym)) return launch_packed(n, kx, X, ldx, scratch, G_hi, G_lo, ldg, gate, st, ctas);
  }
  if (!use_strips(n, kx, sym)) {
    const T* B = sym ? X : Y;
    return launch_one(n, kx, X, ldx, sym ? kx : ky, B, sym ? ldx : ldy, scratch, G_hi, G_lo, ldg, gate, st, ctas, sym, 0,
                      sym);
  }
  for (int c0 = 0; c0 < kx; c0 += 16) {
    const int c1 = std::min(kx, c0 + 16);
    cudaError_t e = launch_one(n, c1, X, ldx, c1 - c0, X + (size_t)c0 * ldx, ldx, scratch, G_hi, G_lo, ldg, gate, st,
                               ctas, true, c0, c0 == 0);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace

// Symmetric: the largest of all forms and of all column counts up to kx, so that
// scratch for the largest of several products holds each of them.
size_t umma_gram_scratch_bytes(int64_t n, int kx, int ky, bool sym) {
  if (sym) ky = kx;
  size_t b = (size_t)num_chunks(n, make_plan(kx, ky, sym)) * (size_t)kx * ky;
  if (!sym) return b * sizeof(FxPart);
  for (int c0 = 0; c0 < kx; c0 += 16) {  // the column strips, one after another
    const int c1 = std::min(kx, c0 + 16);
    b = std::max(b, (size_t)num_chunks(n, make_plan(c1, c1 - c0, c0 == 0)) * (size_t)c1 * (c1 - c0));
  }
  for (int k = 1; k <= std::min(kx, 8); ++k) {  // rows in parts
    const size_t chunks = num_chunks(part_rows_of(n, k), make_plan(k, k, true));
    b = std::max(b, (chunks + 1) * (size_t)k * k);
  }
  return b * sizeof(FxPart);
}

int umma_gram_ctas(int64_t n, int kx, int ky, bool sym, int ctas) {
  if (use_pack(n, kx, sym)) n = part_rows_of(n, kx);
  if (!use_strips(n, kx, sym)) {
    const UPlan plan = make_plan(kx, sym ? kx : ky, sym);
    return plan.nty * capped_chunks(n, plan, ctas);
  }
  int c = 0;
  for (int c0 = 0; c0 < kx; c0 += 16) {
    const int c1 = std::min(kx, c0 + 16);
    const UPlan ps = make_plan(c1, c1 - c0, c0 == 0);
    c = std::max(c, ps.nty * capped_chunks(n, ps, ctas));
  }
  return c;
}

int umma_gram_launches(int64_t n, int kx, const double* X, int64_t ldx, int ky, const double* Y, int64_t ldy,
                       bool sym) {
  (void)X;
  (void)ldx;
  (void)ky;
  (void)Y;
  (void)ldy;
  if (use_pack(n, kx, sym)) return n % (16 * (16 >> pack_lg(kx))) ? 3 : 2;
  return use_strips(n, kx, sym) ? 2 * ((kx + 15) / 16) : 2;
}

cudaError_t launch_umma_gram(int64_t n, int kx, const double* X, int64_t ldx, int ky, const double* Y, int64_t ldy,
                             bool sym, void* scratch, double* G_hi, double* G_lo, int ldg, const int* gate,
                             cudaStream_t st, int ctas) {
  return launch_gram_t<double>(n, kx, X, ldx, ky, Y, ldy, sym, scratch, G_hi, G_lo, ldg, gate, st, ctas);
}

bool umma_gram_f32_supported(const float* X, const float* Y, int kx, int ky, bool sym) {
  (void)kx;
  (void)ky;
  return (uintptr_t)X % 4 == 0 && (sym || (uintptr_t)Y % 4 == 0);
}

cudaError_t launch_umma_gram_f32(int64_t n, int kx, const float* X, int64_t ldx, int ky, const float* Y,
                                 int64_t ldy, bool sym, void* scratch, double* G_hi, double* G_lo, int ldg,
                                 const int* gate, cudaStream_t st) {
  return launch_gram_t<float>(n, kx, X, ldx, ky, Y, ldy, sym, scratch, G_hi, G_lo, ldg, gate, st, 0);
}

}  // namespace eo
