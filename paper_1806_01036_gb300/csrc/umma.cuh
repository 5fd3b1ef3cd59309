// umma.cuh — building blocks of the tcgen05 digit kernels (umma_gram.cu,
// umma_rowprod.cu): inline PTX for mbarriers, TMA, tensor-memory allocation,
// loads and stores, shared-memory matrix descriptors and tcgen05.mma, and the
// 8-bit digits of an FP64 value aligned to a group exponent.
#pragma once

#include <cuda.h>

#include <cstdint>

#include "fx.cuh"

namespace eo {
namespace umma {

using namespace fx;

constexpr unsigned long long kWaitNs = 2000000000ull;  // bound of every mbarrier wait

// ------------------------------------------------------------ PTX helpers
__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned long long gtimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
// One bounded wait: the thread sleeps until the phase completes or up to
// kSuspendNs have passed (no busy polling).
constexpr unsigned kSuspendNs = 1000000u;
__device__ __forceinline__ bool mbar_try_wait(unsigned bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "n"(kSuspendNs)
      : "memory");
  return ok != 0;
}
// Set to 1 by a bounded wait that ran out; the host reads and clears it
// (eo_device_status).  Every translation unit that includes this file has
// its own copy, read through that unit's take_wait_record.
static __device__ unsigned g_wait_expired = 0u;

// Wait for the phase of the given parity to complete.  Gives up (false) once
// *abort is set or after limit_ns, and then sets *abort so that every other
// wait of the CTA gives up at once; a wait that ran out records it in
// g_wait_expired.
static __device__ __noinline__ bool mbar_wait_slow(unsigned bar, unsigned parity, volatile int* abort,
                                                   unsigned long long limit_ns) {
  const unsigned long long t0 = gtimer();
  while (!mbar_try_wait(bar, parity)) {
    const bool late = gtimer() - t0 > limit_ns;
    if (*abort || late) {
      if (late) atomicExch(&g_wait_expired, 1u);
      *abort = 1;
      return false;
    }
  }
  return true;
}
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, volatile int* abort,
                                          unsigned long long limit_ns = kWaitNs) {
  if (mbar_try_wait(bar, parity)) return true;  // the common case: no call
  return mbar_wait_slow(bar, parity, abort, limit_ns);
}
// The same, but only the time limit ends it (waits for MMAs already issued).
static __device__ __noinline__ bool mbar_wait_final(unsigned bar, unsigned parity, volatile int* abort) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = gtimer();
  while (!mbar_try_wait(bar, parity)) {
    if (gtimer() - t0 > kWaitNs) {
      atomicExch(&g_wait_expired, 1u);
      *abort = 1;
      return false;
    }
  }
  return true;
}

// Host side: copy this unit's record to *out (synchronous) and clear it.
static inline cudaError_t take_wait_record(unsigned* out) {
  cudaError_t e = cudaMemcpyFromSymbol(out, g_wait_expired, sizeof(unsigned), 0, cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return e;
  const unsigned zero = 0u;
  return *out ? cudaMemcpyToSymbol(g_wait_expired, &zero, sizeof(unsigned), 0, cudaMemcpyHostToDevice) : e;
}
__device__ __forceinline__ void mbar_arrive(unsigned bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Barrier 1 among the NT threads of the converter warps only, true if any of them passes true.
template <int NT>
__device__ __forceinline__ bool bar_conv_or(bool v) {
  unsigned r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, 1, %2, p;\n selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((unsigned)v), "n"(NT)
      : "memory");
  return r != 0;
}

__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_alloc(unsigned dst, unsigned ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(unsigned taddr, unsigned ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// Shared-memory matrix descriptor: no swizzle, K-major canonical layout;
// lbo = bytes between core matrices adjacent in K, sbo = in M/N.
__device__ __forceinline__ unsigned long long sdesc(unsigned addr, unsigned lbo, unsigned sbo) {
  return (unsigned long long)((addr >> 4) & 0x3fffu) | ((unsigned long long)((lbo >> 4) & 0x3fffu) << 16) |
         ((unsigned long long)((sbo >> 4) & 0x3fffu) << 32) | (1ull << 46);
}
// Instruction descriptor of kind::f16: FP16 A and B (K-major), FP32 D.
__host__ __device__ constexpr unsigned idesc_f16(int M, int N) {
  return (1u << 4) | ((unsigned)(N >> 3) << 17) | ((unsigned)(M >> 4) << 24);
}
__device__ __forceinline__ void mma_f16(unsigned d, unsigned long long a, unsigned long long b, unsigned idesc,
                                        unsigned accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void mma_commit(unsigned bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
               : "memory");
}

// One TMEM column of this warp's 32 lanes (the caller waits).
__device__ __forceinline__ void tmem_ld1(unsigned a, unsigned& v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(v) : "r"(a) : "memory");
}

__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// N consecutive TMEM columns of this warp's 32 lanes (N = 8 or 16).
template <int N>
__device__ __forceinline__ void tmem_ldn(unsigned a, unsigned (&v)[N]) {
  if constexpr (N == 16) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(a)
        : "memory");
  } else {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(a)
                 : "memory");
  }
}
// Completes the loads into v (named, so that no use can move above the wait).
template <int N>
__device__ __forceinline__ void tmem_waitn(unsigned (&v)[N]) {
  if constexpr (N == 16) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                   "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15])
                 :
                 : "memory");
  } else {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7])
                 :
                 : "memory");
  }
}
template <int N>
__device__ __forceinline__ void tmem_stn(unsigned a, const unsigned (&v)[N]) {
  if constexpr (N == 16) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(a),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
        "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
        : "memory");
  } else {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(a), "r"(v[0]), "r"(v[1]),
                 "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
  }
}
template <int N>
__device__ __forceinline__ void tmem_zeron(unsigned a) {
  const unsigned z = 0u;
  if constexpr (N == 16)
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(a),
                 "r"(z)
                 : "memory");
  else
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(a), "r"(z) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// 2-D TMA tile load (box of the tensor map at coordinates (x, y) = (row, column)).
__device__ __forceinline__ void tma_load_2d(unsigned dst, const CUtensorMap* map, int x, int y, unsigned bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          dst),
      "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}

// 3-D box at (x, 0, 0).
__device__ __forceinline__ void tma_load_3d(unsigned dst, const CUtensorMap* map, int x, unsigned bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %3}], [%4];" ::"r"(
          dst),
      "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(0), "r"(bar)
      : "memory");
}

// ------------------------------------------------------------ digits
// A value x aligned to the exponent A of its group (A >= the biased exponent
// of every member) is held as X = floor(|x| 2^(1132 - A)) < 2^110, written with
// 14 balanced base-256 digits, X = sum_s D_s 2^(104 - 8s): the fields of X +
// bias, less 128, D_s in [-128, 127] for s >= 1, and D_0 in [0, 64].  A digit is
// the FP16 integer sign(x) D_s: the field is put into the significand of the FP16 1024
// (bit pattern 0x6400 | f) and one f16x2 FMA takes the offset off and the sign
// on.  Fields are bytes, so two values' digits are cut with one byte
// permutation or one masked merge.  A value within kNearBits binades of A has a
// zero low word, and its digits 10..13 are zero.
constexpr int kNear = 10, kAll = 14;  // digits of a near value, of any value
constexpr int kNearBits = 25;
__device__ __forceinline__ unsigned abs_hi(double x) { return hi32(x) & 0x7fffffffu; }
// Smallest |x| high word of a near value (at least the smallest normal).
__device__ __forceinline__ unsigned near_floor(int A) { return (unsigned)max(A - kNearBits, 1) << 20; }

// X = m 2^t (m the 53-bit significand) as four 32-bit words (w[0] least significant).
__device__ __forceinline__ void any_value_words(double x, int A, unsigned (&w)[4]) {
  const unsigned hi = hi32(x), lo = lo32(x);
  const int e = (hi >> 20) & 0x7ff;
  const unsigned mh = (hi & 0xfffffu) | (e ? 0x100000u : 0u);
  const int t = 57 - A + max(e, 1);
  if (t >= 0) {
    const int bo = t & 31;
    const unsigned s0 = lo << bo, s1 = __funnelshift_l(lo, mh, bo), s2 = __funnelshift_l(mh, 0u, bo);
    const bool up = t >= 32;
    w[0] = up ? 0u : s0;
    w[1] = up ? s0 : s1;
    w[2] = up ? s1 : s2;
    w[3] = up ? s2 : 0u;
  } else {  // more than 52 binades below the column's largest value
    const int r = -t;
    const unsigned long long m = ((unsigned long long)mh << 32) | lo;
    const unsigned long long v = r < 64 ? m >> r : 0ull;
    w[0] = (unsigned)v;
    w[1] = (unsigned)(v >> 32);
    w[2] = 0u;
    w[3] = 0u;
  }
}

// 8-byte asynchronous copy global -> shared; src_bytes 0 writes zeros.
__device__ __forceinline__ void cp_async8z(unsigned dst, const void* src, unsigned src_bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
// 4-byte asynchronous copy global -> shared; src_bytes 0 writes zeros.
__device__ __forceinline__ void cp_async4z(unsigned dst, const void* src, unsigned src_bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit_group() { asm volatile("cp.async.commit_group;" ::: "memory"); }

// The FP16 exponent field of 1024 in both halves, as a register (so that
// the digit's mask and this constant fit one three-input logic operation).
__device__ __forceinline__ unsigned exp1024x2() {
  unsigned r;
  asm volatile("mov.b32 %0, 0x64006400;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned hfma2(unsigned a, unsigned b, unsigned c) {
  unsigned d;
  asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
// Bias of the balanced digits: 128 in each of the digit places 1..13 (bits
// 0..103); the top digit is not negative and takes none.
constexpr unsigned kB = 0x80808080u, kBTop = 0x80u;

// Words 1..3 of X + bias for a value within kNearBits binades of A (X's word 0
// is zero): the significand times 2^bo, bo = t - 32 with X = m 2^t, t = 57 - A
// + e, so bo is in [0, 25].  bo has the sign bit (above the exponent field)
// added as 2^11; shifts take their amount modulo 32.  cA = 25 - A.
// ZERO: a value that is zero gives X = 0 (else the implicit bit would stand).
template <bool ZERO>
__device__ __forceinline__ void near_words(double x, int cA, unsigned& w1, unsigned& w2, unsigned& w3) {
  const unsigned hi = hi32(x), lo = lo32(x);
  const unsigned bo = (hi >> 20) + (unsigned)cA;
  unsigned mh = (hi & 0xfffffu) | 0x100000u;
  if (ZERO) mh = ((hi & 0x7fffffffu) | lo) ? mh : 0u;
  w1 = __funnelshift_l(0u, lo, bo);
  w2 = __funnelshift_l(lo, mh, bo);
  w3 = __funnelshift_l(mh, 0u, bo);
  asm("add.cc.u32 %0, %0, %3;\n\t"
      "addc.cc.u32 %1, %1, %3;\n\t"
      "addc.u32 %2, %2, %4;"
      : "+r"(w1), "+r"(w2), "+r"(w3)
      : "n"(kB), "n"(kBTop));
}

// X + bias of any value (A >= its exponent), four words.
__device__ __forceinline__ void any_words(double x, int A, unsigned (&w)[4]) {
  any_value_words(x, A, w);
  asm("add.cc.u32 %0, %0, %4;\n\t"
      "addc.cc.u32 %1, %1, %4;\n\t"
      "addc.cc.u32 %2, %2, %4;\n\t"
      "addc.u32 %3, %3, %5;"
      : "+r"(w[0]), "+r"(w[1]), "+r"(w[2]), "+r"(w[3])
      : "n"(kB), "n"(kBTop));
}

// f16x2 factors (+-1, +-1) of a pair's digit FMA sign (1024 + f) + addend,
// with the addends -sign 1152 (f - 128) and, for the top digit, -sign 1024.
struct Sign2 {
  unsigned mul, add;
};
__device__ __forceinline__ unsigned hmul2(unsigned a, unsigned b) {
  unsigned d;
  asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ Sign2 sign2(double a, double b) {
  Sign2 s;
  asm("lop3.b32 %0, %1, %2, %3, 0xEA;"
      : "=r"(s.mul)
      : "r"(__byte_perm(hi32(a), hi32(b), 0x7632)), "n"(0x80008000u), "r"(0x3C003C00u));
  s.add = hmul2(s.mul, 0xE480E480u);
  return s;
}
__device__ __forceinline__ Sign2 top(Sign2 s) { return Sign2{s.mul, hmul2(s.mul, 0xE400E400u)}; }
// Both digits of a byte-interleaved lane word z = [lo a, hi a, lo b, hi b].
__device__ __forceinline__ unsigned digit_lo(unsigned z, unsigned e1024, Sign2 s) {
  unsigned f;
  asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(f) : "r"(z), "n"(0x00ff00ffu), "r"(e1024));  // (z & m) | 1024
  return hfma2(f, s.mul, s.add);
}
__device__ __forceinline__ unsigned digit_hi(unsigned z, unsigned e1024, Sign2 s) {
  return hfma2(__byte_perm(z, e1024, 0x7371), s.mul, s.add);  // [z1, 0x64, z3, 0x64]
}


}  // namespace umma
}  // namespace eo
