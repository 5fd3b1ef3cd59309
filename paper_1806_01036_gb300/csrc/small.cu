// small.cu — the k-by-k steps of phase II, one CTA each
// (arXiv:1806.01036, Sec. 4.2: the k-by-k work costs little next to the
// n-row passes, in extended precision too).
//
//   chol_small:  M = R^T R (R upper with positive diagonal) by the
//                square-root-free elimination M = L D L^T, carrying
//                L^{-1} along, so R = D^{1/2} L^T and Z = R^{-1} =
//                L^{-T} D^{-1/2}; T <- R T (R of all passes), and the gates
//                of what follows.
//   svqb_small:  M = U Lambda U^T by cyclic Jacobi in the parallel
//                (round-robin) ordering, Z = U Lambda^{+1/2} U^T = M^{-1/2}
//                (Frobenius-nearest to I among Z with Z^T M Z = I, by the
//                Procrustes argument of the same section), T <- T Z.
//                Rotated form (one pass): the Jacobi runs on D M D with
//                D = diag(M)^{-1/2} and Z = D U Lambda^{+1/2}, columns in
//                ascending eigenvalue order, each eigenvector's largest
//                entry positive (the SVQB of Stathopoulos and Wu, 2002).
// In EO_DD and EO_DD_EFT the arithmetic is floating point with a 128-bit
// significand on the integer pipe (wide.cuh: more accurate than double-double
// and, on this GPU, several times faster), double-double in the pivoted
// Cholesky; otherwise it is FP64.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "wide.cuh"

namespace eo {
namespace {

using namespace fx;

constexpr int kThreads = 256;
constexpr int kJacThreads = 512;
// Jacobi rotates a pair while |a_pq| > eps sqrt(|a_pp a_qq|).  The rotations
// of a sweep leave off-diagonal entries at the rounding level of the
// arithmetic (2^-106 in DD, 2^-53 in FP64), so eps sits a few bits above it:
// at the rounding level itself a sweep would never end without rotations.
constexpr double kJacobiEpsDD = 0x1p-100;
constexpr double kJacobiEpsFP64 = 0x1p-48;

// Double-double (or FP64) arithmetic of the pivoted Cholesky.
template <int MODE>
struct Ar {
  static __device__ __forceinline__ dd sub(dd a, dd b) { return dd{__dsub_rn(a.hi, b.hi), 0.0}; }
  static __device__ __forceinline__ dd mul(dd a, dd b) { return dd{__dmul_rn(a.hi, b.hi), 0.0}; }
  static __device__ __forceinline__ dd sqrt(dd a) { return dd{__dsqrt_rn(a.hi), 0.0}; }
  static __device__ __forceinline__ dd fma(dd a, dd b, dd c) { return dd{__fma_rn(a.hi, b.hi, c.hi), 0.0}; }
  static __device__ __forceinline__ dd recip(dd a) { return dd{__drcp_rn(a.hi), 0.0}; }
};

template <>
struct Ar<MODE_DD> {
  static __device__ __forceinline__ dd sub(dd a, dd b) { return dd_sub(a, b); }
  static __device__ __forceinline__ dd mul(dd a, dd b) { return dd_mul(a, b); }
  static __device__ __forceinline__ dd sqrt(dd a) { return dd_sqrt(a); }
  static __device__ __forceinline__ dd fma(dd a, dd b, dd c) { return dd_add(dd_mul(a, b), c); }
  // 1/a for a > 0: y0 = RN(1/a.hi), whose residual 1 - a.hi y0 is exact in
  // one FMA; with e = 1 - a y0 (|e| <= 2^-52), 1/a = y0 (1 + e + e^2 + ...)
  // and y0 (e + e^2) is the low part (relative error about 2^-105).
  static __device__ __forceinline__ dd recip(dd a) {
    const double y0 = __drcp_rn(a.hi);
    double e = __fma_rn(-a.hi, y0, 1.0);
    e = __fma_rn(-a.lo, y0, e);
    return fast_two_sum(y0, y0 * __fma_rn(e, e, e));
  }
};

__global__ void status_init_kernel(DevStatus* s, int k) {
  for (int i = threadIdx.x; i < 64; i += blockDim.x) s->gate[i] = i == 0;
  if (threadIdx.x == 0) {
    s->info = 0;
    s->rank = k;
    s->iters = 0;
    s->sweeps = 0;
  }
}

__device__ void finish_gates(const SmallGates& g, int run_update, int want_next) {
  *g.upd = run_update;
  if (g.next) *g.next = want_next;
}

// ------------------------------------------------- the two arithmetics

// Vectors of numbers in shared memory, and the operations on them.
struct F64 {
  typedef double T;
  static constexpr size_t kBytes = 8;
  static constexpr bool kLowParts = false;  // a given matrix's low parts are not read
  static constexpr bool kOneSided = false;
  struct Vec {
    double* p;
    __device__ __forceinline__ T get(int i) const { return p[i]; }
    __device__ __forceinline__ void set(int i, T v) const { p[i] = v; }
  };
  // n vectors of the given lengths, one after another
  static __device__ __forceinline__ Vec vec(void* base, size_t total, size_t off) {
    (void)total;
    return Vec{static_cast<double*>(base) + off};
  }
  static __device__ __forceinline__ T zero() { return 0.0; }
  static __device__ __forceinline__ T one() { return 1.0; }
  static __device__ __forceinline__ T neg(T a) { return -a; }
  static __device__ __forceinline__ T from(double hi, double lo) {
    (void)lo;
    return hi;
  }
  static __device__ __forceinline__ void to(T a, double& hi, double& lo) {
    hi = a;
    lo = 0.0;
  }
  static __device__ __forceinline__ T sub(T a, T b) { return __dsub_rn(a, b); }
  static __device__ __forceinline__ T mul(T a, T b) { return __dmul_rn(a, b); }
  static __device__ __forceinline__ T fma(T a, T b, T c) { return __fma_rn(a, b, c); }
  static __device__ __forceinline__ T dot2(T a, T x, T b, T y) { return __dadd_rn(__dmul_rn(a, x), __dmul_rn(b, y)); }
  static __device__ __forceinline__ T recip(T a) { return __drcp_rn(a); }
  static __device__ __forceinline__ T sqrt(T a) { return __dsqrt_rn(a); }
  static __device__ __forceinline__ T rsqrt(T a) { return __ddiv_rn(1.0, __dsqrt_rn(a)); }
  static __device__ __forceinline__ bool is_zero(T a) { return a == 0.0; }
  static __device__ __forceinline__ bool is_neg(T a) { return a < 0.0; }
  static __device__ __forceinline__ bool less(T a, T b) { return a < b; }
  static __device__ __forceinline__ T shfl_xor(T a, int m) { return __shfl_xor_sync(0xffffffffu, a, m); }
  // a pivot that the elimination can divide by (ref: the matrix's own diagonal entry)
  static __device__ __forceinline__ bool pivot_ok(T d, int ref) {
    (void)ref;
    return d > 0.0;
  }
  static __device__ __forceinline__ int scale_of(T a) {
    (void)a;
    return 0;
  }
  // The rotation that zeroes apq: whether |apq| > eps sqrt(|app aqq|), c and s.
  static __device__ __forceinline__ bool rotation(T app, T aqq, T apq, T& c, T& sn) {
    constexpr double eps = kJacobiEpsFP64;
    const double scale = ::sqrt(fabs(app) * fabs(aqq));
    if (!(fabs(apq) > eps * scale && apq != 0.0)) return false;
    const double th = __dsub_rn(aqq, app) / (2.0 * apq);
    const double t = fabs(th) > 1e150 ? 0.5 / th : copysign(1.0 / (fabs(th) + ::sqrt(::fma(th, th, 1.0))), th);
    c = __ddiv_rn(1.0, __dsqrt_rn(__dadd_rn(1.0, __dmul_rn(t, t))));
    sn = __dmul_rn(c, t);
    return true;
  }
};

struct Wide {
  typedef wide T;
  static constexpr bool kLowParts = true;
  static constexpr bool kOneSided = true;  // Jacobi on the Cholesky factor where it can
  static constexpr size_t kBytes = 20;  // significand, exponent and sign in arrays of their own
  struct Vec {
    u128* m;
    int* es;  // 2 e + s
    __device__ __forceinline__ T get(int i) const {
      const int x = es[i];
      return wide{m[i], x >> 1, x & 1};
    }
    __device__ __forceinline__ void set(int i, T v) const {
      m[i] = v.m;
      es[i] = 2 * v.e + v.s;
    }
  };
  static __device__ __forceinline__ Vec vec(void* base, size_t total, size_t off) {
    u128* m = static_cast<u128*>(base);
    return Vec{m + off, reinterpret_cast<int*>(m + total) + off};
  }
  static __device__ __forceinline__ T zero() { return wide_zero(); }
  static __device__ __forceinline__ T one() { return wide_one(); }
  static __device__ __forceinline__ T neg(T a) { return wide_neg(a); }
  static __device__ __forceinline__ T from(double hi, double lo) { return wide_from(hi, lo); }
  static __device__ __forceinline__ void to(T a, double& hi, double& lo) { wide_to_dd(a, hi, lo); }
  static __device__ __forceinline__ T sub(T a, T b) { return wide_sub(a, b); }
  static __device__ __forceinline__ T mul(T a, T b) { return wide_mul(a, b); }
  static __device__ __forceinline__ T fma(T a, T b, T c) { return wide_fma(a, b, c); }
  static __device__ __forceinline__ T dot2(T a, T x, T b, T y) { return wide_dot2(a, x, b, y); }
  static __device__ __forceinline__ T recip(T a) { return wide_recip(a); }
  static __device__ __forceinline__ T sqrt(T a) { return wide_sqrt(a); }
  static __device__ __forceinline__ T rsqrt(T a) { return wide_rsqrt(a); }
  static __device__ __forceinline__ bool is_zero(T a) { return wide_is_zero(a); }
  static __device__ __forceinline__ bool is_neg(T a) { return a.s != 0 && !wide_is_zero(a); }
  static __device__ __forceinline__ bool less(T a, T b) {  // a < b
    const bool na = is_neg(a), nb = is_neg(b);
    return na != nb ? na : (na ? wide_abs_gt(a, b) : wide_abs_gt(b, a));
  }
  static __device__ __forceinline__ T shfl_xor(T a, int m) {
    unsigned long long h = (unsigned long long)(a.m >> 64), l = (unsigned long long)a.m;
    h = __shfl_xor_sync(0xffffffffu, h, m);
    l = __shfl_xor_sync(0xffffffffu, l, m);
    const int x = __shfl_xor_sync(0xffffffffu, 2 * a.e + a.s, m);
    return wide{((u128)h << 64) | l, x >> 1, x & 1};
  }
  // The Gram matrix is given to 2^-106: a pivot 118 binades below its diagonal
  // entry is what rounding left of an exact zero.
  static __device__ __forceinline__ bool pivot_ok(T d, int ref) { return !wide_is_zero(d) && d.s == 0 && d.e > ref - 118; }
  static __device__ __forceinline__ int scale_of(T a) { return a.e; }
  // A rotation: c 2^127 and the tangent +-mt 2^(te - 23), 2^23 <= mt < 2^24.
  struct Turn {
    u128 c;
    unsigned mt;
    int te, s;
  };
  // Leading bits of u 2^(x - 127): f in [1, 2], the binary exponent e.
  static __device__ __forceinline__ void leading(u128 u, int x, float& f, int& e) {
    unsigned long long h = (unsigned long long)(u >> 64), l = (unsigned long long)u;
    if (h == 0ull) {
      h = l;
      l = 0ull;
      x -= 64;
    }
    const int z = clz64(h);
    f = (float)(unsigned)(((h << z) | ((l >> 1) >> (63 - z))) >> 32) * 0x1p-31f;
    e = x - z;
  }
  // Whether |apq| > 2^-100 sqrt(|app aqq|) (leading bits and exponents, all nonzero).
  static __device__ __forceinline__ bool apart(float fpp, int epp, float fqq, int eqq, float fpq, int epq) {
    static_assert(kJacobiEpsDD == 0x1p-100, "the test below");
    const int D = 2 * epq - epp - eqq + 200;  // log2 of apq^2 2^200 / (app aqq), up to the leading bits
    return D >= -2 && (D > 2 || ldexpf(fpq * fpq, D) > fpp * fqq);
  }
  // The rotation that zeroes apq, d = aqq - app: the tangent t from FP32 (24
  // bits: the remainder of apq is left to later sweeps), then c = (1 + t^2)^(-1/2)
  // to 2^-119, so that with s = t c the rotation is orthogonal to that precision.
  static __device__ __forceinline__ Turn turn(float fpq, int epq, int spq, bool dzero, float fd, int ed, int sd) {
    const int x = ed - epq - 1;  // th = d / (2 apq) = +-(fd / fpq) 2^x
    float t;
    int te = 0;  // |t| 2^te
    if (dzero || x < -40) {
      t = 1.0f;
    } else if (x > 40) {
      t = fpq / fd;  // 1 / (2 th)
      te = -x - 1;
    } else {
      const float th = ldexpf(fd / fpq, x);
      t = 1.0f / (th + sqrtf(fmaf(th, th, 1.0f)));
    }
    const float g = te < -20 ? 1.0f : fmaf(ldexpf(t, te), ldexpf(t, te), 1.0f);  // 1 + t^2
    const unsigned bits = __float_as_uint(t);                                       // t in (2^-43, 2)
    const unsigned mt = (bits & 0x7fffffu) | 0x800000u;
    te += (int)(bits >> 23) - 127;
    // 1 + t^2 = G 2^-126: t^2 = mt^2 2^(2 te - 46) (te <= 0, or t = 1 up to its rounding)
    const unsigned long long q = (unsigned long long)mt * mt;
    const int sh = 80 + 2 * te;
    const u128 t2 = sh >= 0 ? (u128)q << sh : shr128((u128)q, -sh);
    return Turn{rsqrt_fixed(((u128)1 << 126) + t2, g), mt, te, dzero ? 0 : sd ^ spq};
  }
  static __device__ __forceinline__ bool rotation(T app, T aqq, T apq, T& c, T& sn) {
    if (wide_is_zero(apq)) return false;
    const float fpq = wide_top(apq);
    if (!apart(wide_top(app), app.e, wide_top(aqq), aqq.e, fpq, apq.e)) return false;
    const wide d = wide_sub(aqq, app);
    const Turn r = turn(fpq, apq.e, apq.s, wide_is_zero(d), wide_top(d), d.e, d.s);
    c = wide_norm(r.c, 0, 0);
    sn = wide_mul(wide{(u128)r.mt << 104, r.te, r.s}, c);
    return true;
  }
};

// Packed upper triangle.
__device__ __forceinline__ int tri(int i, int j) { return j * (j + 1) / 2 + i; }  // i <= j
__device__ __forceinline__ int sym(int i, int j) { return i <= j ? tri(i, j) : tri(j, i); }
__device__ __forceinline__ void untri(int t, int& i, int& j) {  // the entry with tri(i, j) = t
  j = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  if ((j + 1) * (j + 2) / 2 <= t) ++j;
  if (j * (j + 1) / 2 > t) --j;
  i = t - j * (j + 1) / 2;
}

// M's upper triangle into A; false (everywhere) if it has a NaN or Inf (in the parts that are read).  Ends with a barrier.
template <class N>
__device__ __forceinline__ bool load_upper(int k, const double* Mh, const double* Ml, int ldm, typename N::Vec A,
                                           int threads) {
  bool ok = true;
  for (int t = threadIdx.x; t < k * (k + 1) / 2; t += threads) {
    int i, j;
    untri(t, i, j);
    const double h = Mh[(size_t)j * ldm + i], l = N::kLowParts && Ml ? Ml[(size_t)j * ldm + i] : 0.0;
    const bool fin = isfinite(h) && isfinite(l);
    ok = ok && fin;
    A.set(t, fin ? N::from(h, l) : N::zero());
  }
  return __syncthreads_and(ok ? 1 : 0) != 0;
}

// ------------------------------------------------------------ Cholesky

template <class N>
__device__ __forceinline__ void chol_small_body(int k, const double* Mh, const double* Ml, int ldm, SmallWs* ws,
                                                double* Rh_u, double* Rl_u, int ldr, DevStatus* st, SmallGates g,
                                                int pass, int passes, double thr, int* info_user) {
  typedef typename N::T T;
  if (*g.run == 0) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nt = k * (k + 1) / 2;
  // upper triangles: A(i, j), i <= j (becomes R); S, the products of a step;
  // W = L^{-1}, W(l, c) (c <= l) at tri(c, l)
  const typename N::Vec A = N::vec(smem_raw, 3 * (size_t)nt, 0), S = N::vec(smem_raw, 3 * (size_t)nt, nt),
                        W = N::vec(smem_raw, 3 * (size_t)nt, 2 * (size_t)nt);
  __shared__ int flag, ref[KMAX];
  __shared__ double dhi[KMAX];
  __shared__ T piv_inv;
  const int tid = threadIdx.x;
  if (tid == 0) flag = 0;
  if (!load_upper<N>(k, Mh, Ml, ldm, A, kThreads) && tid == 0) flag = -1;
  // Square-root-free (L D L^T) elimination on the upper triangle: at step j
  // the pivot d_j = A(j,j) and the row A(j, j+1..) are those of the
  // standard algorithm before scaling, the Schur complement takes
  // A(a,b) -= A(j,a) A(j,b) / d_j, and W = L^{-1} (L(l,j) = A(j,l) / d_j)
  // takes W(l,:) -= L(l,j) W(j,:).  The products do not depend on the pivot,
  // so they run while one thread forms 1/d_j: the dependent chain of a step
  // is one reciprocal and one multiply-subtract.  Afterwards
  // R = D^{1/2} L^T and Z = R^{-1} = L^{-T} D^{-1/2}.
  for (int t = tid; t < nt; t += kThreads) {
    int i, j;
    untri(t, i, j);
    W.set(t, i == j ? N::one() : N::zero());
    if (i == j) ref[j] = N::scale_of(A.get(t));
  }
  __syncthreads();
  if (flag == 0) {
    for (int j = 0; j < k; ++j) {
      const int m = k - j - 1, np = m * (m + 1) / 2, nq = m * (j + 1);
      if (tid == kThreads - 1) {
        const T d = A.get(tri(j, j));
        if (!N::pivot_ok(d, ref[j])) flag = j + 1;
        else piv_inv = N::recip(d);
      }
      for (int t = tid; t < np + nq; t += kThreads) {
        if (t < np) {  // (a, b) = j + 1 + (u, v), u <= v
          int u, v;
          untri(t, u, v);
          S.set(t, N::mul(A.get(tri(j, j + 1 + u)), A.get(tri(j, j + 1 + v))));
        } else {  // W row l = j + 1 + q % m, column c = q / m <= j
          const int q = t - np, l = j + 1 + q % m, c = q / m;
          S.set(t, N::mul(A.get(tri(j, l)), W.get(tri(c, j))));
        }
      }
      __syncthreads();
      if (flag) break;
      const T w = piv_inv;
      for (int t = tid; t < np + nq; t += kThreads) {
        if (t < np) {
          int u, v;
          untri(t, u, v);
          const int e = tri(j + 1 + u, j + 1 + v);
          A.set(e, N::sub(A.get(e), N::mul(S.get(t), w)));
        } else {
          const int q = t - np, e = tri(q / m, j + 1 + q % m);
          W.set(e, N::sub(W.get(e), N::mul(S.get(t), w)));
        }
      }
      __syncthreads();
    }
  }
  if (flag != 0) {
    if (tid == 0) {
      st->info = flag;
      finish_gates(g, 0, 0);
      if (info_user) *info_user = flag;
    }
    return;
  }
  // s_j = sqrt(d_j) and 1 / s_j (in S(j) for the moment)
  for (int j = tid; j < k; j += kThreads) {
    const T r = N::sqrt(A.get(tri(j, j)));
    A.set(tri(j, j), r);
    S.set(j, N::recip(r));
    double lo;
    N::to(r, dhi[j], lo);
  }
  __syncthreads();
  // R(i, j) = A(i, j) / s_i; Z(i, j) = W(j, i) / s_j (i <= j), straight to memory
  for (int t = tid; t < k * k; t += kThreads) {
    const int i = t % k, j = t / k;
    double h = 0.0, l = 0.0;
    if (i <= j) {
      if (i < j) A.set(tri(i, j), N::mul(A.get(tri(i, j)), S.get(i)));
      N::to(i < j ? N::mul(W.get(tri(i, j)), S.get(j)) : S.get(j), h, l);
    }
    ws->Zh[j * KMAX + i] = h;
    ws->Zl[j * KMAX + i] = l;
  }
  __syncthreads();
  // T <- R T (upper triangular product; the old T into W); T = R on the first pass.
  if (pass != 0) {
    for (int t = tid; t < nt; t += kThreads) {
      int i, j;
      untri(t, i, j);
      W.set(t, N::from(ws->Th[j * KMAX + i], ws->Tl[j * KMAX + i]));
    }
  }
  __syncthreads();
  for (int t = tid; t < k * k; t += kThreads) {
    const int i = t % k, j = t / k;
    double h = 0.0, l = 0.0;
    if (i <= j) {
      T v;
      if (pass == 0) {
        v = A.get(tri(i, j));
      } else {
        v = N::zero();
        for (int q = i; q <= j; ++q) v = N::fma(A.get(tri(i, q)), W.get(tri(q, j)), v);
      }
      N::to(v, h, l);
    }
    ws->Th[j * KMAX + i] = h;
    ws->Tl[j * KMAX + i] = l;
    if (Rh_u) Rh_u[(size_t)j * ldr + i] = h;
    if (Rl_u) Rl_u[(size_t)j * ldr + i] = l;
  }
  if (tid == 0) {
    double dmax = 0.0, dmin = 1e308;
    for (int i = 0; i < k; ++i) {
      dmax = fmax(dmax, dhi[i]);
      dmin = fmin(dmin, dhi[i]);
    }
    int next = 0;
    if (pass == 0) next = passes == 2 ? 1 : (passes == 0 ? (dmax > thr * dmin) : 0);
    finish_gates(g, 1, next);
    if (info_user) *info_user = st->info;
  }
}

// ----------------------------------------- pivoted, partial Cholesky

// One CTA.  A, R and the inverse of R11 in shared memory (double-double in
// EO_DD, FP64 otherwise); see launch_pivchol_small.
template <int MODE>
__global__ void __launch_bounds__(kThreads)
    pivchol_small_kernel(int k, const double* Mh, const double* Ml, int ldm, SmallWs* ws, double* Rh_u,
                         double* Rl_u, int ldr, double tol, DevStatus* st, SmallGates g, int pass, int passes,
                         double thr, int* info_user, int* rank_user, int* perm_user) {
  using A_ = Ar<MODE>;
  if (*g.run == 0) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  dd* A = reinterpret_cast<dd*>(smem_raw);  // A(i,j) = A[j*k+i], the trailing matrix
  dd* R = A + k * k;                        // R(i,j) = R[j*k+i]
  dd* Zs = R + k * k;                       // R11^{-1}
  __shared__ int flag, piv, stop, perm_s[KMAX];
  __shared__ dd rinv;
  const int tid = threadIdx.x;
  const int lim = pass == 0 ? k : st->rank;  // columns that may be factored
  if (tid == 0) {
    flag = 0;
    stop = lim;
  }
  for (int i = tid; i < k; i += kThreads) perm_s[i] = pass == 0 ? i : st->perm[i];
  __syncthreads();
  for (int t = tid; t < k * k; t += kThreads) {
    const int i = t % k, j = t / k;
    const int a = min(i, j), b = max(i, j);
    dd v = dd{Mh[(size_t)b * ldm + a], Ml ? Ml[(size_t)b * ldm + a] : 0.0};
    if (MODE != MODE_DD) v.lo = 0.0;
    if (!dd_finite(v)) atomicExch(&flag, -1);
    A[t] = v;
    R[t] = dd{0.0, 0.0};
    Zs[t] = dd{0.0, 0.0};
  }
  __syncthreads();
  double dmax = 0.0;
  for (int i = 0; i < k; ++i) dmax = fmax(dmax, A[i * k + i].hi);
  const double cut = tol * dmax;
  int r = 0;
  if (flag == 0) {
    for (int j = 0; j < lim; ++j) {
      if (tid == 0) {
        int p = j;
        if (pass == 0)  // the largest remaining diagonal entry, lowest index on ties
          for (int i = j + 1; i < k; ++i) {
            const dd a = A[i * k + i], b = A[p * k + p];
            if (a.hi > b.hi || (a.hi == b.hi && a.lo > b.lo)) p = i;
          }
        const dd d = A[p * k + p];
        if (pass == 0 ? !(d.hi > 0.0 && d.hi > cut) : !(d.hi > 0.0)) {
          stop = j;
          if (pass != 0) flag = j + 1;  // the second pass breaks down
        } else {
          piv = p;
        }
      }
      __syncthreads();
      if (stop == j) break;
      const int p = piv;
      if (p != j) {  // symmetric swap of rows and columns j and p; the rows of R built so far
        for (int i = tid; i < k; i += kThreads) {
          const dd t = A[j * k + i];
          A[j * k + i] = A[p * k + i];
          A[p * k + i] = t;
        }
        __syncthreads();
        for (int i = tid; i < k; i += kThreads) {
          const dd t = A[i * k + j];
          A[i * k + j] = A[i * k + p];
          A[i * k + p] = t;
          if (i < j) {
            const dd u = R[j * k + i];
            R[j * k + i] = R[p * k + i];
            R[p * k + i] = u;
          }
        }
        if (tid == 0) {
          const int t = perm_s[j];
          perm_s[j] = perm_s[p];
          perm_s[p] = t;
        }
        __syncthreads();
      }
      if (tid == 0) {
        const dd rjj = A_::sqrt(A[j * k + j]);
        R[j * k + j] = rjj;
        rinv = A_::recip(rjj);
      }
      __syncthreads();
      for (int l = j + 1 + tid; l < lim; l += kThreads) R[l * k + j] = A_::mul(A[l * k + j], rinv);
      __syncthreads();
      const int m = lim - j - 1;
      for (int t = tid; t < m * m; t += kThreads) {
        const int a = j + 1 + t % m, b = j + 1 + t / m;
        A[b * k + a] = A_::sub(A[b * k + a], A_::mul(R[a * k + j], R[b * k + j]));
      }
      __syncthreads();
      r = j + 1;
    }
  }
  if (flag != 0) {  // NaN / Inf, or a breakdown of the second pass: X stays as it is
    if (tid == 0) {
      st->info = flag;
      if (flag < 0) st->rank = -1;
      finish_gates(g, 0, 0);
      if (info_user) *info_user = flag;
      if (rank_user) *rank_user = st->rank;
    }
    return;
  }
  // R11^{-1}: column c by one thread, back substitution
  for (int c = tid; c < r; c += kThreads) {
    Zs[c * k + c] = A_::recip(R[c * k + c]);
    for (int i = c - 1; i >= 0; --i) {
      dd s2 = dd{0.0, 0.0};
      for (int l = i + 1; l <= c; ++l) s2 = A_::fma(R[l * k + i], Zs[c * k + l], s2);
      Zs[c * k + i] = A_::mul(dd_neg(s2), Zs[i * k + i]);
    }
  }
  __syncthreads();
  // Z: the pivots' rows of R11^{-1} (pass 0), R2^{-1} itself (pass 1); zero beyond the rank
  for (int t = tid; t < KMAX * k; t += kThreads) {
    const int i = t % KMAX, c = t / KMAX;
    if (i < k) {
      ws->Zh[c * KMAX + i] = 0.0;
      ws->Zl[c * KMAX + i] = 0.0;
    }
  }
  __syncthreads();
  for (int t = tid; t < r * r; t += kThreads) {
    const int i = t % r, c = t / r;
    const int row = pass == 0 ? perm_s[i] : i;
    ws->Zh[c * KMAX + row] = Zs[c * k + i].hi;
    ws->Zl[c * KMAX + row] = Zs[c * k + i].lo;
  }
  // R of the whole: R (pass 0) or R2 R_old (pass 1), rows beyond the rank zero
  for (int t = tid; t < k * k; t += kThreads) {
    const int i = t % k, j = t / k;
    dd v = dd{0.0, 0.0};
    if (i < r) {
      if (pass == 0) {
        v = R[j * k + i];
      } else {
        for (int l = i; l < r; ++l) v = A_::fma(R[l * k + i], dd{ws->Th[j * KMAX + l], ws->Tl[j * KMAX + l]}, v);
      }
    }
    Zs[t] = v;
  }
  __syncthreads();
  for (int t = tid; t < k * k; t += kThreads) {
    const int i = t % k, j = t / k;
    ws->Th[j * KMAX + i] = Zs[t].hi;
    ws->Tl[j * KMAX + i] = Zs[t].lo;
    if (Rh_u) Rh_u[(size_t)j * ldr + i] = Zs[t].hi;
    if (Rl_u) Rl_u[(size_t)j * ldr + i] = Zs[t].lo;
  }
  if (pass == 0)
    for (int i = tid; i < k; i += kThreads) {
      st->perm[i] = perm_s[i];
      if (perm_user) perm_user[i] = perm_s[i];
    }
  if (tid == 0) {
    if (pass == 0) st->rank = r;
    int next = 0;
    if (pass == 0 && r > 0)
      next = passes == 2 ? 1 : (passes == 0 ? (R[0].hi > thr * R[(r - 1) * k + (r - 1)].hi) : 0);
    finish_gates(g, 1, next);
    if (info_user) *info_user = st->info;
    if (rank_user) *rank_user = st->rank;
  }
}

// ------------------------------------------------- one-sided Jacobi

// x c >> 128 for signed x and 0 <= c < 2^128 (below the exact value by at most 3).
__device__ __forceinline__ i128 smulhi128(i128 x, u128 c) {
  return (i128)(mulhi128((u128)x, c) - (x < 0 ? c : (u128)0));
}
__device__ __forceinline__ i128 sar128(i128 x, int n) {  // n >= 0
  return n < 127 ? x >> n : (x < 0 ? (i128)-1 : (i128)0);
}
__device__ __forceinline__ i128 shfl_sum(i128 v) {  // over the warp
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) {
    const unsigned long long h = __shfl_xor_sync(0xffffffffu, (unsigned long long)((u128)v >> 64), m);
    const unsigned long long l = __shfl_xor_sync(0xffffffffu, (unsigned long long)(u128)v, m);
    v += (i128)(((u128)h << 64) | l);
  }
  return v;
}
// v 2^x as a wide number
__device__ __forceinline__ wide wide_int(i128 v, int x) {
  const bool neg = v < 0;
  return wide_norm(neg ? (u128)-v : (u128)v, x + 127, neg ? 1 : 0);
}
// A column of up to 32 NQ entries, NQ per lane, in units 2^(E - 125): shifted so
// that its largest magnitude lies in [2^121, 2^122) (so that its norm is below
// 2^125); from units 2^x.  Returns E.
template <int NQ>
__device__ __forceinline__ int settle(i128 (&v)[NQ], int x) {
  auto top = [](i128 a) { return (unsigned)((u128)(a < 0 ? ~a : a) >> 95); };
  auto low = [](i128 a) { return (unsigned)((u128)(a < 0 ? ~a : a) >> 63); };
  unsigned t = __reduce_max_sync(0xffffffffu, max(top(v[0]), top(v[NQ - 1])));
  int z;
  if (t) {
    z = __clz((int)t) - 5;  // |largest| in [2^(126 - clz), 2^(127 - clz))
  } else {
    t = __reduce_max_sync(0xffffffffu, max(low(v[0]), low(v[NQ - 1])));
    z = t ? __clz((int)t) + 27 : 59;  // (a column that cancels further is settled again by its next rotation)
  }
#pragma unroll
  for (int q = 0; q < NQ; ++q) v[q] = z >= 0 ? (i128)((u128)v[q] << z) : v[q] >> -z;
  return x - z + 125;
}

// v mt 2^-24, mt < 2^24, rounded down.
__device__ __forceinline__ i128 smul24(i128 v, unsigned mt) {
  const i128 h = (i128)(long long)(v >> 64) * (long long)mt;
  const u128 l = (u128)(unsigned long long)v * mt;
  return (i128)((u128)h << 40) + (i128)(l >> 24);
}

// One warp makes two columns of up to 32 NQ entries (units 2^(ex - 125) and
// 2^(ey - 125)) orthogonal; false if they already are.  With s = t c the columns
// become c (x - t y) and c (y + t x): t has 24 bits, so a product by t is a
// quarter of a product by c.
template <int NQ>
__device__ __forceinline__ bool rotate_pair(int k, i128* wx, i128* wy, int& Ex, int& Ey, int lane) {
  i128 x[NQ], y[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int i = lane + 32 * q;
    x[q] = i < k ? wx[i] : (i128)0;
    y[q] = i < k ? wy[i] : (i128)0;
  }
  const int ex = Ex, ey = Ey;
  // sums of squares and products, units 2^(2 E - 250 + 128)
  i128 sxx = 0, syy = 0, sxy = 0;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const u128 ax = (u128)(x[q] < 0 ? -x[q] : x[q]), ay = (u128)(y[q] < 0 ? -y[q] : y[q]);
    sxx += (i128)mulhi128(ax, ax);
    syy += (i128)mulhi128(ay, ay);
    const i128 m = (i128)mulhi128(ax, ay);
    sxy += (x[q] < 0) != (y[q] < 0) ? -m : m;
  }
  sxx = shfl_sum(sxx);
  syy = shfl_sum(syy);
  sxy = shfl_sum(sxy);
  if (sxy == 0 || sxx == 0 || syy == 0) return false;
  float fxx, fyy, fxy, fd;
  int exx, eyy, exy, ed;
  Wide::leading((u128)sxx, 2 * ex - 122, fxx, exx);
  Wide::leading((u128)syy, 2 * ey - 122, fyy, eyy);
  Wide::leading((u128)(sxy < 0 ? -sxy : sxy), ex + ey - 122, fxy, exy);
  if (!Wide::apart(fxx, exx, fyy, eyy, fxy, exy)) return false;
  // the difference in the units of the larger exponent
  const int top = max(ex, ey);
  const i128 d = (i128)shr128((u128)syy, 2 * (top - ey)) - (i128)shr128((u128)sxx, 2 * (top - ex));
  Wide::leading((u128)(d < 0 ? -d : d), 2 * top - 122, fd, ed);
  const Wide::Turn r = Wide::turn(fxy, exy, sxy < 0 ? 1 : 0, d == 0, fd, ed, d < 0 ? 1 : 0);
  // t y and t x in units 2^(E + te - 124); the columns in units 2^(mx - 125), 2^(my - 125) before the product by c / 2
  const int mx = max(ex, ey + r.te + 1), my = max(ey, ex + r.te + 1);
  i128 nx[NQ], ny[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const i128 ty = sar128(smul24(y[q], r.mt), mx - ey - r.te - 1), tx = sar128(smul24(x[q], r.mt), my - ex - r.te - 1);
    nx[q] = smulhi128(sar128(x[q], mx - ex) + (r.s ? ty : -ty), r.c);
    ny[q] = smulhi128(sar128(y[q], my - ey) + (r.s ? -tx : tx), r.c);
  }
  const int fx = settle(nx, mx - 124), fy = settle(ny, my - 124);
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int i = lane + 32 * q;
    if (i < k) {
      wx[i] = nx[q];
      wy[i] = ny[q];
    }
  }
  __syncwarp();
  if (lane == 0) {
    Ex = fx;
    Ey = fy;
  }
  return true;
}

// Eigenvalues and vectors of a positive semidefinite M (A, packed; destroyed) by
// one-sided Jacobi on its Cholesky factor with diagonal pivoting (Drmac and
// Veselic): M = L L^T, and rotations V that make the columns of L V orthogonal
// give the eigenvectors as its normalized columns, their squared norms as the
// eigenvalues (into A's diagonal; zero for the columns beyond the rank).
// Against the two-sided form on M it needs about half the sweeps on a graded
// spectrum, no second matrix to update, and no exponent per entry: a column is
// 128-bit fixed point with one exponent (errors 2^-118 of its norm).  One warp
// takes a pair of columns through a whole rotation (three sums over the rows,
// the angle, the update), so that a step has one barrier.  Bound by the issue of
// its integer instructions, one CTA on one SM: about 1000 a warp and step (2000
// with products by sine and cosine in 128 bits and the angle on wide numbers).
// SVQB step of k = 32: about 10 ms with double-doubles on the FP64 pipe, 1.35 in
// this form, 0.95 with the 24-bit tangent.
// False (with M's triangle to be loaded again) when M is not semidefinite to
// rounding (a row that is dropped keeps an entry above 2^-100 of the diagonal's
// scale, or its diagonal entry is negative by more), or its diagonal spans more than 100 binades, where small entries
// need exponents of their own.
__device__ bool onesided_jacobi(int k, const Wide::Vec A, const Wide::Vec U, DevStatus* st) {
  __shared__ int E[KMAX], ref[KMAX], pos[KMAX], col[KMAX];
  __shared__ wide inv;
  __shared__ int piv, state, rot_count;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < k) {
    ref[tid] = A.get(tri(tid, tid)).e;
    pos[tid] = k;  // step at which the row was eliminated
    col[tid] = -1;  // row eliminated at a step (-1: none)
  }
  if (tid == 0) state = 0;
  __syncthreads();
  {
    int lo = 1 << 30, hi = -(1 << 30);  // exponents of the nonzero diagonal entries
    for (int i = lane; i < k; i += 32) {
      if (ref[i] == kWideZero) continue;
      lo = min(lo, ref[i]);
      hi = max(hi, ref[i]);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (hi - lo > 100) return false;
  }
  // M = L L^T in the order of the largest remaining diagonal entries: column
  // `step` of L is A(:, p) / sqrt(d) over the rows not eliminated before.  An
  // entry that rounding alone may have left is dropped (no column).
  for (int step = 0; step < k; ++step) {
    if (warp == 0) {
      unsigned long long best = 0;  // exponent and leading bits, then the index from the top
      for (int i = lane; i < k; i += 32) {
        if (pos[i] != k) continue;
        const wide d = A.get(tri(i, i));
        const bool good = !wide_is_zero(d) && d.s == 0;
        const unsigned long long key = good ? ((unsigned long long)(unsigned)(d.e + (1 << 29)) << 32) |
                                                  ((unsigned)(d.m >> 96) & ~63u) | (unsigned)(63 - i)
                                            : (unsigned long long)(63 - i) + 1;
        best = key > best ? key : best;
      }
#pragma unroll
      for (int m = 16; m >= 1; m >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, best, m);
        best = o > best ? o : best;
      }
      const bool good = best >> 32;
      const int p = 63 - (int)((good ? best : best - 1) & 63ull);
      const wide d = A.get(tri(p, p));
      const bool ok = good && Wide::pivot_ok(d, ref[p]);
      if (!ok) {
        // nothing left of the row but rounding?  (of a semidefinite M a diagonal
        // entry of zero leaves a row of zeros)
        bool rest = false;
        for (int i = lane; i < k; i += 32) {
          if (pos[i] != k || i == p) continue;
          const wide a = A.get(sym(i, p));
          rest |= !wide_is_zero(a) && 2 * a.e > ref[i] + ref[p] - 200;
        }
        if (__any_sync(0xffffffffu, rest) && lane == 0) state = 1;
      }
      if (lane == 0) {
        piv = ok ? p : -1;
        pos[p] = step;
        if (ok) {
          inv = wide_recip(d);
          col[step] = p;
        } else if (d.s && !wide_is_zero(d) && d.e > ref[p] - 100) {
          state = 1;  // a negative diagonal entry: not semidefinite
        }
      }
    }
    __syncthreads();
    if (state) return false;
    const int p = piv;
    if (p >= 0) {
      const wide w = inv;
      for (int t = tid; t < k * (k + 1) / 2; t += kJacThreads) {
        int a, b;
        untri(t, a, b);
        if (pos[a] == k && pos[b] == k)
          A.set(t, wide_sub(A.get(t), wide_mul(wide_mul(A.get(sym(a, p)), w), A.get(sym(b, p)))));
      }
    }
    __syncthreads();
  }
  // L's columns in fixed point, rows in M's order (U's significands)
  i128* W = reinterpret_cast<i128*>(U.m);
  for (int l = warp; l < k; l += kJacThreads / 32) {
    const int p = col[l];
    wide x[2] = {wide_zero(), wide_zero()};
    if (p >= 0) {
      const wide r = wide_rsqrt(A.get(tri(p, p)));
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int i = lane + 32 * q;
        if (i < k && pos[i] >= l) x[q] = wide_mul(A.get(sym(i, p)), r);
      }
    }
    const int top = __reduce_max_sync(0xffffffffu, max(x[0].e, x[1].e));
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int i = lane + 32 * q;
      const i128 v = (i128)shr128(x[q].m, p >= 0 ? min(128, 6 + top - x[q].e) : 128);
      if (i < k) W[l * k + i] = x[q].s ? -v : v;
    }
    if (lane == 0) E[l] = p >= 0 ? top + 4 : 0;
  }
  __syncthreads();
  const int kk = k + (k & 1), npairs = kk / 2;
  for (int sweep = 0; sweep < 40; ++sweep) {
    if (tid == 0) rot_count = 0;
    __syncthreads();
    for (int step = 0; step < kk - 1; ++step) {
      for (int pr = warp; pr < npairs; pr += kJacThreads / 32) {
        // round-robin pairing: player 0 fixed, the others rotate by `step`
        auto player = [&](int at) { return at == 0 ? 0 : 1 + (at - 1 + step) % (kk - 1); };
        const int a = player(pr), b = player(kk - 1 - pr);
        const int lo = min(a, b), hi = max(a, b);
        if (hi >= k) continue;
        if (k <= 32 ? rotate_pair<1>(k, W + lo * k, W + hi * k, E[lo], E[hi], lane)
                    : rotate_pair<2>(k, W + lo * k, W + hi * k, E[lo], E[hi], lane)) {
          if (lane == 0) atomicAdd(&rot_count, 1);
        }
      }
      __syncthreads();
    }
    if (rot_count == 0) {
      if (tid == 0) st->sweeps = sweep + 1;
      break;
    }
    __syncthreads();
    if (sweep == 39 && tid == 0) st->sweeps = 40;
  }
  // eigenvalues and normalized columns
  for (int l = warp; l < k; l += kJacThreads / 32) {
    i128 x[2], sxx = 0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int i = lane + 32 * q;
      x[q] = i < k ? W[l * k + i] : (i128)0;
      const u128 ax = (u128)(x[q] < 0 ? -x[q] : x[q]) << 2;  // (a norm below 2^127)
      sxx += (i128)mulhi128(ax, ax);
    }
    const wide lam = wide_int(shfl_sum(sxx), 2 * E[l] - 126);
    const wide r = wide_is_zero(lam) ? wide_zero() : wide_rsqrt(lam);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int i = lane + 32 * q;
      if (i < k) U.set(l * k + i, wide_mul(wide_int(x[q], E[l] - 125), r));
    }
    if (lane == 0) A.set(tri(l, l), lam);
  }
  __syncthreads();
  return true;
}

// --------------------------------------------------------------- SVQB

template <class N>
__device__ __forceinline__ void svqb_small_body(int k, const double* Mh, const double* Ml, int ldm, SmallWs* ws,
                                                double* Zh_u, double* Zl_u, int ldz, double tol, DevStatus* st,
                                                SmallGates g, int pass, int passes, double thr, int* rank_user,
                                                bool rotated) {
  typedef typename N::T T;
  if (*g.run == 0) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nt = k * (k + 1) / 2;
  const int kk = k + (k & 1);  // even number of players; index k is a dummy
  const int npairs = kk / 2;
  // A and the next A (upper triangles), U (columns), c and s per pair, D = diag(M)^{-1/2} (rotated form)
  const size_t total = 2 * (size_t)nt + (size_t)k * k + 2 * (size_t)npairs + k;
  typename N::Vec A = N::vec(smem_raw, total, 0), A2 = N::vec(smem_raw, total, nt);
  const typename N::Vec U = N::vec(smem_raw, total, 2 * (size_t)nt),
                        cs = N::vec(smem_raw, total, 2 * (size_t)nt + (size_t)k * k),
                        dv = N::vec(smem_raw, total, 2 * (size_t)nt + (size_t)k * k + 2 * (size_t)npairs);
  __shared__ int pr[KMAX + 2];   // p, q per pair
  __shared__ int perm[KMAX];     // eigenpair of column j (rotated form)
  __shared__ int rotates[KMAX / 2 + 1];
  __shared__ int rot_count, next_unit;
  const int tid = threadIdx.x, lane = tid & 31;
  if (!load_upper<N>(k, Mh, Ml, ldm, A, kJacThreads)) {
    if (tid == 0) {
      st->rank = -1;
      finish_gates(g, 0, 0);
      if (rank_user) *rank_user = -1;
    }
    return;
  }
  if (rotated) {  // the Jacobi runs on D M D (unit diagonal; a zero diagonal gives d_i = 0)
    for (int i = tid; i < k; i += kJacThreads) {
      const T m = A.get(tri(i, i));
      dv.set(i, !N::is_zero(m) && !N::is_neg(m) ? N::rsqrt(m) : N::zero());
      perm[i] = i;
    }
    __syncthreads();
    for (int t = tid; t < nt; t += kJacThreads) {
      int i, j;
      untri(t, i, j);
      A.set(t, N::mul(N::mul(dv.get(i), A.get(t)), dv.get(j)));
    }
  }
  __syncthreads();
  auto twosided = [&]() {
    // Sweeps of the parallel (round-robin) ordering.  Per step: (1) each pair's
    // rotation (N::rotation: the angle in a short format, c and s orthogonal to
    // full precision; the remainder of a_pq is removed by later sweeps); (2) A' =
    // J^T A J by 2x2 blocks of pairs on the upper triangle, into the second
    // buffer, and U <- U J in place.  The warps take units of (2) from a counter:
    // first 16 blocks a unit (a pair of lanes per block: each multiplies a row by
    // J_Q, then, after an exchange, a column by J_P^T), then 64 entries of U.
    const int nblk = npairs * (npairs + 1) / 2, ablk = (nblk + 15) / 16, uent = 2 * npairs * k, nunits = ablk + (uent + 63) / 64;
    for (int sweep = 0; sweep < 40; ++sweep) {
      if (tid == 0) rot_count = 0;
      __syncthreads();
      for (int step = 0; step < kk - 1; ++step) {
        // round-robin pairing: player 0 fixed, the others rotate by `step`
        if (tid < npairs) {
          auto player = [&](int pos) { return pos == 0 ? 0 : 1 + (pos - 1 + step) % (kk - 1); };
          const int a = player(tid), b = player(kk - 1 - tid);
          const int lo = min(a, b), hi = max(a, b);
          T c = N::one(), sn = N::zero();
          const bool rot = hi < k && N::rotation(A.get(tri(lo, lo)), A.get(tri(hi, hi)), A.get(tri(lo, hi)), c, sn);
          if (rot) atomicAdd(&rot_count, 1);
          rotates[tid] = rot;
          cs.set(2 * tid, c);
          cs.set(2 * tid + 1, sn);
          pr[2 * tid] = lo;
          pr[2 * tid + 1] = hi;
        }
        if (tid == kJacThreads - 1) next_unit = 0;
        __syncthreads();
        for (;;) {
          int unit = 0;
          if (lane == 0) unit = atomicAdd(&next_unit, 1);
          unit = __shfl_sync(0xffffffffu, unit, 0);
          if (unit >= nunits) break;
          if (unit < ablk) {
            // A2 = J^T A J, block (P, Q) of rows {lo_P, hi_P} and columns {lo_Q, hi_Q}, P <= Q
            const int b = unit * 16 + (lane >> 1), r = lane & 1;
            const bool act = b < nblk;
            int P, Q;
            untri(act ? b : 0, P, Q);
            const int r0 = pr[2 * P], r1 = pr[2 * P + 1], c0 = pr[2 * Q], c1 = pr[2 * Q + 1];
            const bool v1 = r1 < k, w1 = c1 < k;  // r0, c0 < k always (the dummy index is the larger)
            const int row = r ? r1 : r0;
            const bool have = !r || v1;
            T t0 = have ? A.get(sym(row, c0)) : N::zero();
            T t1 = have && w1 ? A.get(sym(row, c1)) : N::zero();
            if (rotates[Q]) {  // row r of B J_Q
              const T c = cs.get(2 * Q), sn = cs.get(2 * Q + 1);
              const T x = N::dot2(t0, c, t1, N::neg(sn));
              t1 = N::dot2(t0, sn, t1, c);
              t0 = x;
            }
            const T other = N::shfl_xor(r ? t0 : t1, 1);
            T y0 = r ? other : t0, y1 = r ? t1 : other;  // column r
            if (rotates[P]) {  // J_P^T (B J_Q)
              const T c = cs.get(2 * P), sn = cs.get(2 * P + 1);
              const T x = N::dot2(c, y0, N::neg(sn), y1);
              y1 = N::dot2(sn, y0, c, y1);
              y0 = x;
            }
            if (act && (!r || w1)) {
              const int col = r ? c1 : c0;
              A2.set(sym(r0, col), y0);
              if (v1 && (P != Q || r)) A2.set(sym(r1, col), y1);  // (P = Q: (r1, c0) is the mirror of (r0, c1))
            }
          } else {
            // U <- U J, columns lo_Q, hi_Q of row m: a pair of lanes per row and pair
            for (int h = 0; h < 2; ++h) {
              const int t = (unit - ablk) * 64 + h * 32 + lane;
              const int q = (t >> 1) / k, m = (t >> 1) % k, r = t & 1;
              const bool act = t < uent && rotates[q] != 0;
              T v = N::zero();
              if (act) {
                const T c = cs.get(2 * q), sn = cs.get(2 * q + 1);
                const T x = U.get(pr[2 * q] * k + m), y = U.get(pr[2 * q + 1] * k + m);
                v = r ? N::dot2(sn, x, c, y) : N::dot2(c, x, N::neg(sn), y);
              }
              __syncwarp();  // both lanes have read the entries that they replace
              if (act) U.set(pr[2 * q + r] * k + m, v);
            }
          }
        }
        __syncthreads();
        const typename N::Vec sw = A;
        A = A2;
        A2 = sw;
      }
      if (rot_count == 0) {
        if (tid == 0) st->sweeps = sweep + 1;
        break;
      }
      __syncthreads();
      if (sweep == 39 && tid == 0) st->sweeps = 40;
    }
  };
  // M itself (or D M D) is kept in A2 in case the one-sided form declines it
  bool done = false;
  if constexpr (N::kOneSided) {
    for (int t = tid; t < nt; t += kJacThreads) A2.set(t, A.get(t));
    __syncthreads();
    done = onesided_jacobi(k, A, U, st);
    if (!done) {
      __syncthreads();
      const typename N::Vec sw = A;
      A = A2;
      A2 = sw;
    }
  }
  if (!done) {
    for (int t = tid; t < k * k; t += kJacThreads) U.set(t, t % k == t / k ? N::one() : N::zero());
    __syncthreads();
    twosided();
  }
  if (rotated) {
    // Column a of U: its largest-magnitude entry (lowest row on ties) made
    // positive; its place in the ascending order of the eigenvalues (ties by
    // index) gives the column of Z it lands in.
    auto mag = [](T x) { return N::is_neg(x) ? N::neg(x) : x; };
    for (int a = tid; a < k; a += kJacThreads) {
      int mb = 0;
      T best = mag(U.get(a * k));
      for (int m = 1; m < k; ++m) {
        const T x = mag(U.get(a * k + m));
        if (N::less(best, x)) {
          best = x;
          mb = m;
        }
      }
      if (N::is_neg(U.get(a * k + mb)))
        for (int m = 0; m < k; ++m) U.set(a * k + m, N::neg(U.get(a * k + m)));
      const T la = A.get(tri(a, a));
      int pos = 0;
      for (int b = 0; b < k; ++b) {
        const T lb = A.get(tri(b, b));
        pos += N::less(lb, la) || (!N::less(la, lb) && b < a);
      }
      perm[pos] = a;  // pos < k; with a NaN eigenvalue two columns may collide, the rest keep the identity
    }
    __syncthreads();
  }
  // w_l = lambda_l^{-1/2} for kept eigenvalues (in cs, which has at least k entries)
  __shared__ double lam[KMAX];
  __shared__ double lmax_s, lmin_s;
  __shared__ int rank_s;
  for (int i = tid; i < k; i += kJacThreads) {
    double lo;
    N::to(A.get(tri(i, i)), lam[i], lo);
  }
  __syncthreads();
  if (tid == 0) {
    double lmax = 0.0;
    for (int i = 0; i < k; ++i) lmax = lam[i] > lmax ? lam[i] : lmax;
    const double cut = tol * lmax;
    int rank = 0;
    double lmin = lmax;
    for (int i = 0; i < k; ++i)
      if (lmax > 0.0 && lam[i] > cut) {
        ++rank;
        lmin = lam[i] < lmin ? lam[i] : lmin;
      }
    lmax_s = lmax;
    lmin_s = lmin;
    rank_s = rank;
  }
  __syncthreads();
  for (int i = tid; i < k; i += kJacThreads)
    cs.set(i, lmax_s > 0.0 && lam[i] > tol * lmax_s ? N::rsqrt(A.get(tri(i, i))) : N::zero());
  __syncthreads();
  auto out_z = [&](int i, int j, T v, bool last) {  // Z, and T = Z when there is no earlier transform
    double h, l;
    N::to(v, h, l);
    ws->Zh[j * KMAX + i] = h;
    ws->Zl[j * KMAX + i] = l;
    if (!last) return;
    ws->Th[j * KMAX + i] = h;
    ws->Tl[j * KMAX + i] = l;
    if (Zh_u) Zh_u[(size_t)j * ldz + i] = h;
    if (Zl_u) Zl_u[(size_t)j * ldz + i] = l;
  };
  if (rotated) {  // Z(:, j) = D u_a w_a with a = perm[j] (one pass)
    for (int t = tid; t < k * k; t += kJacThreads) {
      const int i = t % k, j = t / k, a = perm[j];
      out_z(i, j, N::mul(N::mul(dv.get(i), U.get(a * k + i)), cs.get(a)), true);
    }
  } else {
    // Z = U diag(w) U^T = (U diag(w)^{1/2}) (U diag(w)^{1/2})^T: one triangle,
    // mirrored, so that Z is exactly symmetric (into A2)
    for (int t = tid; t < k * k; t += kJacThreads) U.set(t, N::mul(U.get(t), N::sqrt(cs.get(t / k))));
    __syncthreads();
    for (int t = tid; t < nt; t += kJacThreads) {
      int i, j;
      untri(t, i, j);
      T v = N::zero();
      for (int l = 0; l < k; ++l) v = N::fma(U.get(l * k + i), U.get(l * k + j), v);
      A2.set(t, v);
      out_z(i, j, v, pass == 0);
      if (i != j) out_z(j, i, v, pass == 0);
    }
    if (pass != 0) {  // T <- T Z (the old T into U)
      __syncthreads();
      for (int t = tid; t < k * k; t += kJacThreads) {
        const size_t e = (size_t)(t / k) * KMAX + t % k;
        U.set(t, N::from(ws->Th[e], ws->Tl[e]));
      }
      __syncthreads();
      for (int t = tid; t < k * k; t += kJacThreads) {
        const int i = t % k, j = t / k;
        T v = N::zero();
        for (int l = 0; l < k; ++l) v = N::fma(U.get(l * k + i), A2.get(sym(l, j)), v);
        double h, lo;
        N::to(v, h, lo);
        ws->Th[j * KMAX + i] = h;
        ws->Tl[j * KMAX + i] = lo;
        if (Zh_u) Zh_u[(size_t)j * ldz + i] = h;
        if (Zl_u) Zl_u[(size_t)j * ldz + i] = lo;
      }
    }
  }
  if (tid == 0) {
    st->rank = rank_s;
    int next = 0;
    if (pass == 0) next = passes == 2 ? 1 : (passes == 0 ? (lmax_s > thr * thr * lmin_s) : 0);
    finish_gates(g, 1, next);
    if (rank_user) *rank_user = rank_s;
  }
}

// ----------------------------------------------------- kernel wrappers

template <int MODE>
using Num = std::conditional_t<MODE == MODE_DD, Wide, F64>;

template <int MODE>
__global__ void __launch_bounds__(kThreads) chol_small_kernel(int k, const double* Mh, const double* Ml, int ldm,
                                                              SmallWs* ws, double* Rh_u, double* Rl_u, int ldr,
                                                              DevStatus* st, SmallGates g, int pass, int passes,
                                                              double thr, int* info_user) {
  chol_small_body<Num<MODE>>(k, Mh, Ml, ldm, ws, Rh_u, Rl_u, ldr, st, g, pass, passes, thr, info_user);
}

template <int MODE>
__global__ void __launch_bounds__(kJacThreads, 1) svqb_small_kernel(int k, const double* Mh, const double* Ml, int ldm,
                                                              SmallWs* ws, double* Zh_u, double* Zl_u, int ldz,
                                                              double tol, DevStatus* st, SmallGates g, int pass,
                                                              int passes, double thr, int* rank_user,
                                                              bool rotated) {
  svqb_small_body<Num<MODE>>(k, Mh, Ml, ldm, ws, Zh_u, Zl_u, ldz, tol, st, g, pass, passes, thr, rank_user, rotated);
}

// One CTA per job: the factorization of pass `pass` of many independent
// blocks, each from its own workspace's Gram matrix and gates.
__device__ __forceinline__ SmallGates job_gates(const SmallJob& j, int pass, int npass) {
  return SmallGates{&j.st->gate[2 * pass], &j.st->gate[2 * pass + 1],
                    pass + 1 < npass ? &j.st->gate[2 * pass + 2] : nullptr};
}

template <int MODE>
__global__ void __launch_bounds__(kThreads) chol_small_batched_kernel(const SmallJob* jobs, int pass, int passes,
                                                                      double thr) {
  const SmallJob j = jobs[blockIdx.x];
  const int npass = passes == 1 ? 1 : 2;
  chol_small_body<Num<MODE>>(j.k, j.ws->Mh, j.ws->Ml, KMAX, j.ws, j.Oh, j.Ol, j.ldo, j.st, job_gates(j, pass, npass), pass,
                        passes, thr, j.out);
}

template <int MODE>
__global__ void __launch_bounds__(kJacThreads, 1) svqb_small_batched_kernel(const SmallJob* jobs, int pass, int passes,
                                                                      double thr) {
  const SmallJob j = jobs[blockIdx.x];
  const int npass = passes == 1 ? 1 : 2;
  svqb_small_body<Num<MODE>>(j.k, j.ws->Mh, j.ws->Ml, KMAX, j.ws, j.Oh, j.Ol, j.ldo, j.tol, j.st,
                        job_gates(j, pass, npass), pass, passes, thr, j.out, false);
}

__global__ void status_init_batched_kernel(const SmallJob* jobs, int njobs) {
  for (int b = blockIdx.x; b < njobs; b += gridDim.x) {
    DevStatus* s = jobs[b].st;
    for (int i = threadIdx.x; i < 64; i += blockDim.x) s->gate[i] = i == 0;
    if (threadIdx.x == 0) {
      s->info = 0;
      s->rank = jobs[b].k;
      s->iters = 0;
      s->sweeps = 0;
    }
  }
}

// ------------------------------------------------------ convergence test

__global__ void __launch_bounds__(kThreads) converge_kernel(const int* run, const double* Ch, const double* Cl, int ldc,
                                                            int kv, int k, const double* Mh, const double* Ml,
                                                            int ldm, double eps, DevStatus* st, int iter,
                                                            int max_iter, int* iters_user, int* rank_user) {
  if (*run == 0) return;
  // Frobenius norms of C and of M - I (each bounds the 2-norm from above),
  // as sums of squares in a fixed reduction order
  __shared__ double red[2][kThreads];
  double sc = 0.0, sm = 0.0;
  for (int t = threadIdx.x; t < kv * k; t += kThreads) {
    const int i = t % kv, j = t / kv;
    const double c = Ch[(size_t)j * ldc + i] + (Cl ? Cl[(size_t)j * ldc + i] : 0.0);
    sc += c * c;
  }
  for (int t = threadIdx.x; t < k * k; t += kThreads) {
    const int i = t % k, j = t / k;
    // (M_hi - delta) + M_lo: the subtraction of 1 is exact near 1
    const double e = (Mh[(size_t)j * ldm + i] - (i == j ? 1.0 : 0.0)) + (Ml ? Ml[(size_t)j * ldm + i] : 0.0);
    sm += e * e;
  }
  red[0][threadIdx.x] = sc;
  red[1][threadIdx.x] = sm;
  __syncthreads();
  for (int w = kThreads / 2; w >= 1; w >>= 1) {
    if (threadIdx.x < w) {
      red[0][threadIdx.x] += red[0][threadIdx.x + w];
      red[1][threadIdx.x] += red[1][threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double fc = sqrt(red[0][0]), fm = sqrt(red[1][0]);
    const bool conv = fc <= eps && fm <= eps;  // false for NaN
    st->gate[kItSvqb + iter] = conv ? 0 : 1;
    if (iter + 1 < max_iter) st->gate[kItRun + iter + 1] = conv ? 0 : 1;
    if (conv) st->iters = iter;  // updates applied before convergence was seen
    else if (iter + 1 == max_iter) st->iters = -max_iter;
    if (iters_user && (conv || iter + 1 == max_iter)) *iters_user = st->iters;
    if (rank_user && conv) *rank_user = st->rank;  // k when no SVQB was needed
  }
}

}  // namespace

cudaError_t launch_converge(const int* run, const double* Ch, const double* Cl, int ldc, int kv, int k,
                            const double* Mh, const double* Ml, int ldm, double eps, DevStatus* s, int iter,
                            int max_iter, int* iters_user, int* rank_user, cudaStream_t st) {
  converge_kernel<<<1, kThreads, 0, st>>>(run, Ch, Cl, ldc, kv, k, Mh, Ml, ldm, eps, s, iter, max_iter, iters_user,
                                          rank_user);
  return cudaGetLastError();
}

__global__ void symmetrize_kernel(int k, double* Mh, double* Ml, int ld, const int* gate) {
  if (gate && *gate == 0) return;
  for (int t = threadIdx.x; t < k * k; t += blockDim.x) {
    const int i = t % k, j = t / k;
    if (i >= j) continue;  // one thread per pair i < j
    const size_t u = (size_t)j * ld + i, l = (size_t)i * ld + j;
    dd s = dd_add(dd{Mh[u], Ml ? Ml[u] : 0.0}, dd{Mh[l], Ml ? Ml[l] : 0.0});
    s.hi *= 0.5;  // halving is exact
    s.lo *= 0.5;
    Mh[u] = Mh[l] = s.hi;
    if (Ml) Ml[u] = Ml[l] = s.lo;
  }
}

cudaError_t launch_symmetrize(int k, double* Mh, double* Ml, int ld, const int* gate, cudaStream_t st) {
  symmetrize_kernel<<<1, 256, 0, st>>>(k, Mh, Ml, ld, gate);
  return cudaGetLastError();
}

cudaError_t launch_status_init(DevStatus* s, int k, cudaStream_t st) {
  status_init_kernel<<<1, 32, 0, st>>>(s, k);
  return cudaGetLastError();
}

size_t pivchol_smem(int k) { return 3 * (size_t)k * k * sizeof(dd); }
size_t chol_smem(bool wide, int k) { return 3 * (size_t)(k * (k + 1) / 2) * (wide ? Wide::kBytes : F64::kBytes); }
size_t svqb_smem(bool wide, int k) {
  const size_t n = (size_t)k * (k + 1) + (size_t)k * k + 2 * (size_t)((k + 1) / 2) + k;
  return n * (wide ? Wide::kBytes : F64::kBytes);
}

cudaError_t launch_pivchol_small(Mode mode, int k, const double* Mh, const double* Ml, int ldm, SmallWs* ws,
                                 double* R_hi, double* R_lo, int ldr, double tol, DevStatus* s, SmallGates g,
                                 int pass, int passes, int* info_user, int* rank_user, int* perm_user,
                                 cudaStream_t st) {
  const size_t smem = pivchol_smem(k);
  cudaError_t e;
  if (mode == MODE_DD) {
    e = set_dyn_smem(pivchol_small_kernel<MODE_DD>, smem);
    if (e != cudaSuccess) return e;
    pivchol_small_kernel<MODE_DD><<<1, kThreads, smem, st>>>(k, Mh, Ml, ldm, ws, R_hi, R_lo, ldr, tol, s, g, pass,
                                                              passes, 1e7, info_user, rank_user, perm_user);
  } else {
    e = set_dyn_smem(pivchol_small_kernel<MODE_FP64>, smem);
    if (e != cudaSuccess) return e;
    pivchol_small_kernel<MODE_FP64><<<1, kThreads, smem, st>>>(k, Mh, Ml, ldm, ws, R_hi, R_lo, ldr, tol, s, g,
                                                                pass, passes, 1e4, info_user, rank_user, perm_user);
  }
  return cudaGetLastError();
}
cudaError_t launch_chol_small(Mode mode, int k, const double* Mh, const double* Ml, int ldm, SmallWs* ws,
                              double* R_hi, double* R_lo, int ldr, DevStatus* s, SmallGates g, int pass, int passes,
                              int* info_user, cudaStream_t st) {
  const size_t smem = chol_smem(mode == MODE_DD, k);
  cudaError_t e;
  if (mode == MODE_DD) {
    e = set_dyn_smem(chol_small_kernel<MODE_DD>, smem);
    if (e != cudaSuccess) return e;
    chol_small_kernel<MODE_DD><<<1, kThreads, smem, st>>>(k, Mh, Ml, ldm, ws, R_hi, R_lo, ldr, s, g, pass, passes,
                                                         1e7, info_user);
  } else {
    e = set_dyn_smem(chol_small_kernel<MODE_FP64>, smem);
    if (e != cudaSuccess) return e;
    chol_small_kernel<MODE_FP64><<<1, kThreads, smem, st>>>(k, Mh, Ml, ldm, ws, R_hi, R_lo, ldr, s, g, pass, passes,
                                                           1e4, info_user);
  }
  return cudaGetLastError();
}

cudaError_t launch_svqb_small(Mode mode, int k, const double* Mh, const double* Ml, int ldm, SmallWs* ws,
                              double* Z_hi, double* Z_lo, int ldz, double tol, DevStatus* s, SmallGates g, int pass,
                              int passes, int* rank_user, cudaStream_t st, bool rotated) {
  const size_t smem = svqb_smem(mode == MODE_DD, k);
  if (rotated) passes = 1;
  cudaError_t e;
  if (mode == MODE_DD) {
    if (tol < 0) tol = k * 0x1p-104;
    e = set_dyn_smem(svqb_small_kernel<MODE_DD>, smem);
    if (e != cudaSuccess) return e;
    svqb_small_kernel<MODE_DD><<<1, kJacThreads, smem, st>>>(k, Mh, Ml, ldm, ws, Z_hi, Z_lo, ldz, tol, s, g, pass,
                                                         passes, 1e7, rank_user, rotated);
  } else {
    if (tol < 0) tol = k * 0x1p-52;
    e = set_dyn_smem(svqb_small_kernel<MODE_FP64>, smem);
    if (e != cudaSuccess) return e;
    svqb_small_kernel<MODE_FP64><<<1, kJacThreads, smem, st>>>(k, Mh, Ml, ldm, ws, Z_hi, Z_lo, ldz, tol, s, g, pass,
                                                           passes, 1e4, rank_user, rotated);
  }
  return cudaGetLastError();
}

double svqb_default_tol(Mode mode, int k) { return mode == MODE_DD ? k * 0x1p-104 : k * 0x1p-52; }

cudaError_t launch_status_init_batched(const SmallJob* jobs, int njobs, cudaStream_t st) {
  status_init_batched_kernel<<<std::min(njobs, 1024), 64, 0, st>>>(jobs, njobs);
  return cudaGetLastError();
}

cudaError_t launch_small_batched(bool chol, Mode mode, int njobs, int kmax, const SmallJob* jobs, int pass,
                                 int passes, cudaStream_t st) {
  const bool ddm = mode == MODE_DD;
  cudaError_t e;
  if (chol) {
    const size_t smem = chol_smem(ddm, kmax);
    auto kern = ddm ? chol_small_batched_kernel<MODE_DD> : chol_small_batched_kernel<MODE_FP64>;
    e = set_dyn_smem(kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<njobs, kThreads, smem, st>>>(jobs, pass, passes, ddm ? 1e7 : 1e4);
  } else {
    // A DD Jacobi eigensolve of 16 or more columns fills most of an SM's issue
    // slots on its own (a k = 32 one takes 1 ms alone): when several share
    // an SM they all slow down and the launch ends with the last of them.
    // Asking for more than half of an SM's shared memory keeps one such CTA
    // per SM (the jobs are ordered widest first, so the first wave spreads
    // the widest over the SMs).
    size_t smem = svqb_smem(ddm, kmax);
    if (kmax >= 16) smem = std::max<size_t>(smem, 116 * 1024);
    auto kern = ddm ? svqb_small_batched_kernel<MODE_DD> : svqb_small_batched_kernel<MODE_FP64>;
    e = set_dyn_smem(kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<njobs, kJacThreads, smem, st>>>(jobs, pass, passes, ddm ? 1e7 : 1e4);
  }
  return cudaGetLastError();
}

}  // namespace eo
