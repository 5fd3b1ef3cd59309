// update.cu — the final multiplication Y = Y~ Z of phase II
// (arXiv:1806.01036, Sec. 4.2: the multiplication by Z that ends phase II; CholQR uses
// the upper-triangular Z = R^{-1}, SVQB the full symmetric Z).
//
// Each thread owns whole rows: it loads the k entries of its row, then forms
// q_j = sum_i x_i Z_ij (i <= j for triangular Z) with DD accumulation of the
// exact products x_i * (Z_hi + Z_lo)_ij in EO_DD (one rounding per entry), or
// FP64 fma accumulation otherwise.  All loads of a row precede its stores, so
// the update is done in place.  Z lives in shared memory.
#include <algorithm>

#include "common.cuh"

namespace eo {
namespace {

constexpr int kThreads = 128;
// FP32 blocks of 9 to 32 columns run on the tensor-core digits from 16384 rows
// on: exact sums rounded once, where the loop below is bound by the FP64 pipe.
// One CholQR pass with this kernel and with the digits, 2e6 rows: 8 columns
// 632 vs 562 us, 9 1219 vs 815, 16 1398 vs 503, 32 5944 vs 1318; 20,000 rows:
// 8 59 vs 57 us, 9 73 vs 67, 32 182 vs 168; below, the digits' start costs what
// they save (1e4 rows, 16 columns: 73 vs 75).  (The digits' groups of more than
// 32 columns would need scratch that the FP32 mode does not reserve.)
bool f32_digits(int64_t n, int k) { return k >= 9 && k <= 32 && n >= 16384; }

// Bound by the FP64 pipe (2 FMA a clock and SM).  TRI: the triangle written out
// (k <= KM <= 32, FP64 accumulation).  A loop whose FMAs past the diagonal are
// predicated off spends the pipe's time on them all the same: 500,000 x 16, one
// update, 240 -> 118 us (its FMAs alone: 116).  The sums keep their order.
template <int MODE, typename T, int KM, bool TRI>
__global__ void __launch_bounds__(kThreads) update_kernel(int64_t n, int k, T* X, int64_t ldx,
                                                          const double* __restrict__ Zh, const double* __restrict__ Zl,
                                                          int tri, const int* gate) {
  if (gate && *gate == 0) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  dd* Zs = reinterpret_cast<dd*>(smem_raw);  // k-by-k, leading dimension k
  for (int t = threadIdx.x; t < k * k; t += kThreads) {
    const int i = t % k, j = t / k;
    Zs[j * k + i] = dd{Zh[(size_t)j * KMAX + i], Zl[(size_t)j * KMAX + i]};
  }
  __syncthreads();
  const int64_t stride = (int64_t)gridDim.x * kThreads;
  for (int64_t r = (int64_t)blockIdx.x * kThreads + threadIdx.x; r < n; r += stride) {
    double x[KM];  // the whole row stays in registers, so q_j may overwrite x_j at once
#pragma unroll
    for (int i = 0; i < KM; ++i) x[i] = i < k ? (double)X[(size_t)i * ldx + r] : 0.0;
    if constexpr (TRI) {
#pragma unroll
      for (int j = 0; j < KM; ++j) {
        if (j >= k) break;
        double s = 0.0;
#pragma unroll
        for (int i = 0; i <= j; ++i) s = __fma_rn(x[i], Zs[j * k + i].hi, s);
        X[(size_t)j * ldx + r] = (T)s;
      }
    } else {
#pragma unroll 1
      for (int j = 0; j < k; ++j) {
        const int iend = tri ? j + 1 : k;
        double q;
        if (MODE == MODE_DD) {
          dd s = dd{0.0, 0.0};
#pragma unroll
          for (int i = 0; i < KM; ++i)
            if (i < iend) dd_fma_acc_dd(s, Zs[j * k + i], x[i]);
          q = __dadd_rn(s.hi, s.lo);
        } else {
          double s = 0.0;
#pragma unroll
          for (int i = 0; i < KM; ++i)
            if (i < iend) s = __fma_rn(x[i], Zs[j * k + i].hi, s);
          q = s;
        }
        X[(size_t)j * ldx + r] = (T)q;
      }
    }
  }
}

template <int MODE, typename T>
cudaError_t launch_k(int64_t n, int k, void* X, int64_t ldx, const double* Zh, const double* Zl, bool tri,
                     const int* gate, cudaStream_t st) {
  T* x = static_cast<T*>(X);
  int64_t blocks64 = (n + kThreads - 1) / kThreads;
  int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(blocks64, 152 * 16));
  const int t = tri ? 1 : 0;
  const size_t smem = (size_t)k * k * sizeof(dd);
  cudaError_t e = cudaSuccess;
  constexpr bool kTri = MODE != MODE_DD;
  if (k <= 8) {
    if (kTri && tri) update_kernel<MODE, T, 8, kTri><<<blocks, kThreads, smem, st>>>(n, k, x, ldx, Zh, Zl, t, gate);
    else update_kernel<MODE, T, 8, false><<<blocks, kThreads, smem, st>>>(n, k, x, ldx, Zh, Zl, t, gate);
  } else if (k <= 16) {
    if (kTri && tri) update_kernel<MODE, T, 16, kTri><<<blocks, kThreads, smem, st>>>(n, k, x, ldx, Zh, Zl, t, gate);
    else update_kernel<MODE, T, 16, false><<<blocks, kThreads, smem, st>>>(n, k, x, ldx, Zh, Zl, t, gate);
  } else if (k <= 32) {
    if (kTri && tri) update_kernel<MODE, T, 32, kTri><<<blocks, kThreads, smem, st>>>(n, k, x, ldx, Zh, Zl, t, gate);
    else update_kernel<MODE, T, 32, false><<<blocks, kThreads, smem, st>>>(n, k, x, ldx, Zh, Zl, t, gate);
  } else {
    e = set_dyn_smem(update_kernel<MODE, T, 64, false>, smem);
    if (e != cudaSuccess) return e;
    update_kernel<MODE, T, 64, false><<<blocks, kThreads, smem, st>>>(n, k, x, ldx, Zh, Zl, t, gate);
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_update(Mode mode, int64_t n, int k, void* X, int64_t ldx, const double* Zh, const double* Zl,
                          bool tri, const int* gate, cudaStream_t st) {
  switch (mode) {
    case MODE_DD: return launch_k<MODE_DD, double>(n, k, X, ldx, Zh, Zl, tri, gate, st);
    case MODE_F32:
      if (f32_digits(n, k))
        return launch_umma_update_f32(n, k, static_cast<float*>(X), ldx, Zh, Zl, KMAX, tri, gate, st);
      return launch_k<MODE_F32, float>(n, k, X, ldx, Zh, Zl, tri, gate, st);
    default: return launch_k<MODE_FP64, double>(n, k, X, ldx, Zh, Zl, tri, gate, st);
  }
}

}  // namespace eo
