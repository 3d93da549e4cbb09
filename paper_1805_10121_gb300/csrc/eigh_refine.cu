// The projected eigenproblem G = W diag(lambda) W^H at FP64 accuracy from an
// FP32 eigensolve.
//
// Why.  FP64 runs 64 times narrower than FP32 here, and the dense eigensolver
// of the vendor's library, the largest part of a Rayleigh-Ritz step, takes
// 4.1 ms (p = 70) or 8.5 ms (p = 197) in FP64 against 1.3 and 2.0 ms in FP32.
// Products at FP64 accuracy are cheap (rns.cu), and a refinement made of
// products alone doubles the correct digits per step (Ogita and Aishima,
// "Iterative refinement for symmetric eigenvalue decomposition", JJIAM 2018):
// with X the approximate eigenvectors,
//
//   S = X^H G X,  M = X^H X,  lambda_i = S_ii / M_ii,
//   E_ij = (S_ij - (lambda_i + lambda_j) M_ij / 2) / (lambda_j - lambda_i) - M_ij / 2,
//   E_ii = (1 - M_ii) / 2,   X <- X + X E,
//
// to ||E||_F <= 1e-8, after which the next correction is below rounding: three
// or four steps of about 0.1 ms.  G is shifted by its mean diagonal and scaled
// first, so the FP32 solve resolves the spread of the spectrum, not its place.
//
// Close eigenvalues.  A numerator at rounding level is no reason to rotate
// (degenerate pairs): E_ij = -M_ij / 2 keeps the columns orthonormal.  Where
// the quotient is not small, FP32 could not tell the two directions apart, and
// the pair is rotated exactly (a Jacobi rotation) before the next step.  Too
// many such pairs, or no convergence in eight steps, and the caller takes the
// FP64 eigensolver on the untouched G.
#include <algorithm>
#include <cmath>
#include <numeric>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "context.hpp"

namespace chase {
namespace {

constexpr int kThreads = 256;
constexpr int kMaxPairs = 64;  // pairs rotated between two steps
constexpr double kRotate = 0.1;  // |E_ij| from which a pair is rotated

template <class T>
struct Elem;
template <>
struct Elem<chase_c64> {
  using D = double2;
  using F = float2;
  using Single = chase_c32;
};
template <>
struct Elem<double> {
  using D = double;
  using F = float;
  using Single = float;
};

__device__ __forceinline__ double re(double2 a) { return a.x; }
__device__ __forceinline__ double re(double a) { return a; }
__device__ __forceinline__ double abs2(double2 a) { return a.x * a.x + a.y * a.y; }
__device__ __forceinline__ double abs2(double a) { return a * a; }
__device__ __forceinline__ double2 axpy(double2 y, double f, double2 x) {  // y + f x
  return make_double2(fma(f, x.x, y.x), fma(f, x.y, y.y));
}
__device__ __forceinline__ double axpy(double y, double f, double x) { return fma(f, x, y); }
__device__ __forceinline__ double2 times(double2 a, double f) { return make_double2(a.x * f, a.y * f); }
__device__ __forceinline__ double times(double a, double f) { return a * f; }
__device__ __forceinline__ double2 mul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double mul(double a, double b) { return a * b; }
__device__ __forceinline__ double2 conj(double2 a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ double conj(double a) { return a; }
__device__ __forceinline__ void shift_diag(double2& a, double c) {
  a.x -= c;
  a.y = 0.0;
}
__device__ __forceinline__ void shift_diag(double& a, double c) { a -= c; }
__device__ __forceinline__ float2 narrow(double2 a, double f) {
  return make_float2(static_cast<float>(a.x * f), static_cast<float>(a.y * f));
}
__device__ __forceinline__ float narrow(double a, double f) { return static_cast<float>(a * f); }

__device__ double block_sum(double v, double* scratch) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = v;
  __syncthreads();
  v = 0.0;
#pragma unroll
  for (int w = 0; w < kThreads / 32; ++w) v += scratch[w];
  return v;
}

// What a step reports to the host.
struct Report {
  double centre;      // mean diagonal of G
  int npairs, pad;
  int pair[kMaxPairs][2];
};

// A = G - c I, c the mean diagonal, and the norm of each column of A.
template <class D>
__global__ void __launch_bounds__(kThreads)
    centre_kernel(const D* __restrict__ G, long long ldg, int p, D* __restrict__ A, long long lda,
                  double* __restrict__ norm, Report* __restrict__ rep) {
  __shared__ double scratch[kThreads / 32];
  double c = 0.0;
  for (int i = threadIdx.x; i < p; i += kThreads) c += re(G[i * ldg + i]);
  c = block_sum(c, scratch) / p;
  const int j = blockIdx.x;
  if (j == 0 && threadIdx.x == 0) rep->centre = c;
  double s = 0.0;
  for (int i = threadIdx.x; i < p; i += kThreads) {
    D v = G[j * ldg + i];
    if (i == j) shift_diag(v, c);
    A[j * lda + i] = v;
    s += abs2(v);
  }
  s = block_sum(s, scratch);
  if (threadIdx.x == 0) norm[j] = sqrt(s);
}

// The power of two that scales A to a largest column norm in [1, 2), and the
// scaled ||A||_F^2; one warp, the result in all its lanes.
__device__ __forceinline__ double column_scale(const double* __restrict__ norm, int p, double* f2) {
  const int lane = threadIdx.x & 31;
  double m = 0.0, s = 0.0;
  for (int i = lane; i < p; i += 32) m = fmax(m, norm[i]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  int e = 0;
  if (m > 0.0) frexp(m, &e);
  const double f = ldexp(1.0, max(-1000, min(1000, 1 - e)));
  for (int i = lane; i < p; i += 32) s = fma(norm[i] * f, norm[i] * f, s);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  *f2 = s;
  return f;
}

// F = A scaled by a power of two to a largest column norm in [1, 2).
template <class D, class F>
__global__ void __launch_bounds__(kThreads)
    narrow_kernel(const D* __restrict__ A, long long lda, int p, const double* __restrict__ norm,
                  F* __restrict__ out, long long ldo) {
  __shared__ double s_f;
  if (threadIdx.x < 32) {
    double f2;
    const double f = column_scale(norm, p, &f2);
    if (threadIdx.x == 0) s_f = f;
  }
  __syncthreads();
  const double f = s_f;
  const int j = blockIdx.x;
  for (int i = threadIdx.x; i < p; i += kThreads) out[j * ldo + i] = narrow(A[j * lda + i], f);
}

// ---------------------------------------------------------------------------
// The FP32 solve up to p = 96: one-sided Jacobi in one block's shared memory.
// With A' = A + c I, c = ||A||_F, positive definite, rotations that make the
// columns of B = A' J orthogonal turn J into eigenvectors and each column of B
// into a multiple of one, so J itself is not needed.  A warp holds a pair of
// columns in registers; the p / 2 pairs of a round are disjoint, and p - 1
// rounds meet every pair (round robin).  Latency bounds it, 1.4 us a round: dot
// product, rotation and the block's barrier.  The library's solver, hundreds of
// launches of a few microseconds, takes 1.3 ms at p = 70 whatever G is; here a
// dense G takes about as long (eigensolve in all 2.1 ms on either; p = 33: 0.82
// against 1.34 ms; whole Rayleigh-Ritz call, N = 1000: 2.04 ms at p = 96 here,
// 2.22 at p = 97 with the library), one near a diagonal, as from the second
// iteration of a solve on, 0.6 ms.
// ---------------------------------------------------------------------------
constexpr int kJacobiMax = 96, kJacobiThreads = 1024;
constexpr int kJacobiSweeps = 14;

__device__ __forceinline__ void add_diag(float2& a, float v) { a.x += v; }
__device__ __forceinline__ void add_diag(float& a, float v) { a += v; }
__device__ __forceinline__ float2 conj_dot(float2 acc, float2 a, float2 b) {  // acc + conj(a) b
  return make_float2(fmaf(a.x, b.x, fmaf(a.y, b.y, acc.x)), fmaf(a.x, b.y, fmaf(-a.y, b.x, acc.y)));
}
__device__ __forceinline__ float conj_dot(float acc, float a, float b) { return fmaf(a, b, acc); }
__device__ __forceinline__ float norm2(float2 a) { return fmaf(a.x, a.x, a.y * a.y); }
__device__ __forceinline__ float norm2(float a) { return a * a; }
__device__ __forceinline__ float2 cmul_conj(float2 a, float2 e) {  // a conj(e)
  return make_float2(fmaf(a.x, e.x, a.y * e.y), fmaf(a.y, e.x, -a.x * e.y));
}
__device__ __forceinline__ float cmul_conj(float a, float e) { return a * e; }
__device__ __forceinline__ float2 scale_f(float2 a, float f) { return make_float2(a.x * f, a.y * f); }
__device__ __forceinline__ float scale_f(float a, float f) { return a * f; }
__device__ __forceinline__ float2 combine(float2 a, float c, float2 b, float s) {  // c a + s b
  return make_float2(fmaf(c, a.x, s * b.x), fmaf(c, a.y, s * b.y));
}
__device__ __forceinline__ float combine(float a, float c, float b, float s) {
  return fmaf(c, a, s * b);
}
__device__ __forceinline__ float warp_add(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// The two parts in the two halves of the warp after the first exchange: seven
// shuffles instead of ten.
__device__ __forceinline__ float2 warp_add(float2 v) {
  const bool upper = threadIdx.x & 16;
  float a = upper ? v.y : v.x;
  a += __shfl_xor_sync(0xffffffffu, upper ? v.x : v.y, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  const float b = __shfl_xor_sync(0xffffffffu, a, 16);
  return upper ? make_float2(b, a) : make_float2(a, b);
}
__device__ __forceinline__ double2 widen(float2 a, float f) {
  return make_double2(static_cast<double>(a.x) * f, static_cast<double>(a.y) * f);
}
__device__ __forceinline__ double widen(float a, float f) { return static_cast<double>(a) * f; }

// R: rows of a column per lane, p <= 32 R.
template <int R, class D, class F>
__global__ void __launch_bounds__(kJacobiThreads, 1)
    jacobi_kernel(const D* __restrict__ A, long long lda, int p, const double* __restrict__ norm,
                  D* __restrict__ X, long long ldx) {
  extern __shared__ double jacobi_smem[];
  F* B = reinterpret_cast<F*>(jacobi_smem);  // p x p, column-major
  __shared__ int s_rotated[2];
  __shared__ float s_norm[kJacobiMax];  // squared column norms
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int kWarps = kJacobiThreads / 32;
  __shared__ double s_f;
  __shared__ float s_shift;
  if (warp == 0) {
    double f2;  // ||A||_F^2 of the scaled matrix
    const double f = column_scale(norm, p, &f2);
    if (lane == 0) {
      s_f = f;
      s_shift = fmaxf(1.0625f * sqrtf(static_cast<float>(f2)), 1.f);
    }
  }
  __syncthreads();
  const double f = s_f;
  const float shift = s_shift;
  for (int q = threadIdx.x; q < p * p; q += kJacobiThreads) {
    const int i = q % p, j = q / p;
    F v = narrow(A[j * lda + i], f);
    if (i == j) add_diag(v, shift);
    B[q] = v;
  }
  if (threadIdx.x < 2) s_rotated[threadIdx.x] = 0;
  __syncthreads();
  const int n = (p + 1) & ~1;
  for (int sweep = 0; sweep < kJacobiSweeps; ++sweep) {
    // afresh in each sweep; a rotation moves t |g| between the two
    for (int j = warp; j < p; j += kWarps) {
      float v = 0.f;
      for (int i = lane; i < p; i += 32) v += norm2(B[j * p + i]);
      v = warp_add(v);
      if (lane == 0) s_norm[j] = v;
    }
    __syncthreads();
    for (int round = 0; round < n - 1; ++round) {
      for (int k = warp; k < n / 2; k += kWarps) {
        const int k2 = n - 1 - k;
        const int i = k == 0 ? 0 : 1 + (k - 1 + round) % (n - 1);
        const int j = 1 + (k2 - 1 + round) % (n - 1);
        if (i >= p || j >= p) continue;
        F a[R], b[R], g = F{};
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int row = lane + 32 * r;
          a[r] = row < p ? B[i * p + row] : F{};
          b[r] = row < p ? B[j * p + row] : F{};
          g = conj_dot(g, a[r], b[r]);
        }
        const float na = s_norm[i], nb = s_norm[j];
        g = warp_add(g);
        const float g2 = norm2(g);
        // cosine below FP32's resolution: orthogonal
        if (!(g2 > 4e-14f * na * nb)) continue;
        const float ig = rsqrtf(g2);
        const F ph = scale_f(g, ig);
        const float zeta = 0.5f * (nb - na) * ig;
        const float t =
            copysignf(__fdividef(1.f, fabsf(zeta) + sqrtf(fmaf(zeta, zeta, 1.f))), zeta);
        const float c = rsqrtf(fmaf(t, t, 1.f)), s = t * c;
        __syncwarp();  // every lane has read both norms
        if (lane == 0) {
          const float move = t * g2 * ig;
          s_norm[i] = na - move;
          s_norm[j] = nb + move;
          if (g2 > 1e-12f * na * nb) s_rotated[sweep & 1] = 1;
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int row = lane + 32 * r;
          const F h = cmul_conj(b[r], ph);
          if (row < p) {
            B[i * p + row] = combine(a[r], c, h, -s);
            B[j * p + row] = combine(a[r], s, h, c);
          }
        }
      }
      __syncthreads();
    }
    const int rotated = s_rotated[sweep & 1];
    if (threadIdx.x == 0) s_rotated[(sweep + 1) & 1] = 0;
    __syncthreads();
    if (!rotated) break;
  }
  for (int j = warp; j < p; j += kWarps) {
    float s = 0.f;
    for (int i = lane; i < p; i += 32) s += norm2(B[j * p + i]);
    s = rsqrtf(warp_add(s));
    for (int i = lane; i < p; i += 32) X[j * ldx + i] = widen(B[j * p + i], s);
  }
}

// Column j of E, its squared norm, the eigenvalues, and the pairs to rotate.
template <class D>
__global__ void __launch_bounds__(kThreads)
    correction_kernel(const D* __restrict__ S, const D* __restrict__ M, long long ld, int p,
                      const double* __restrict__ norm, D* __restrict__ E,
                      double* __restrict__ lambda, double* __restrict__ e2, Report* __restrict__ rep) {
  extern __shared__ double lam[];
  __shared__ double scratch[kThreads / 32];
  double a2 = 0.0;
  for (int i = threadIdx.x; i < p; i += kThreads) {
    lam[i] = re(S[i * ld + i]) / re(M[i * ld + i]);
    a2 = fma(norm[i], norm[i], a2);
  }
  // numerators that rounding alone explains: a few units of ||A||_F
  const double noise = 4.0 * 1.1102230246251565e-16 * sqrt(block_sum(a2, scratch));
  const int j = blockIdx.x;
  const double lj = lam[j];
  if (j == 0)
    for (int i = threadIdx.x; i < p; i += kThreads) lambda[i] = lam[i];
  double s = 0.0;
  for (int i = threadIdx.x; i < p; i += kThreads) {
    const D m = M[j * ld + i];
    D e = times(m, -0.5);
    if (i == j) {
      shift_diag(e, -0.5);
    } else {
      // anti-Hermitian: one triangle of S and one test for both (i, j) and
      // (j, i), or E + E^H = I - M and with it X's orthonormality is lost
      const D sij = i < j ? S[j * ld + i] : conj(S[i * ld + j]);
      const D k = axpy(sij, -0.5 * (lj + lam[i]), m);
      const double gap = lj - lam[i], n = sqrt(abs2(k));
      if (!(n <= noise)) {
        if (n <= kRotate * fabs(gap)) {
          e = axpy(e, 1.0 / gap, k);
        } else if (i < j) {
          const int q = atomicAdd(&rep->npairs, 1);
          if (q < kMaxPairs) {
            rep->pair[q][0] = i;
            rep->pair[q][1] = j;
          }
        }
      }
    }
    E[j * ld + i] = e;
    s += abs2(e);
  }
  s = block_sum(s, scratch);
  if (threadIdx.x == 0) e2[j] = s;
}

// Columns (i, k) of X and S, and rows of S, by the rotation that makes S_ik
// zero; the pairs in their order (one block).
struct Pairs {
  int n;
  int pair[kMaxPairs][2];
};
template <class D>
__global__ void __launch_bounds__(kThreads)
    rotate_kernel(D* __restrict__ S, D* __restrict__ X, long long ld, int p,
                  const __grid_constant__ Pairs pairs) {
  for (int q = 0; q < pairs.n; ++q) {
    const int i = pairs.pair[q][0], k = pairs.pair[q][1];
    const double a = re(S[i * ld + i]), b = re(S[k * ld + k]);
    const D s = S[k * ld + i];
    const double r = sqrt(abs2(s));
    __syncthreads();
    if (!(r > 0.0)) continue;
    const double tau = (b - a) / (2.0 * r);
    const double t = copysign(1.0, tau) / (fabs(tau) + sqrt(fma(tau, tau, 1.0)));
    const double c = 1.0 / sqrt(fma(t, t, 1.0)), sn = t * c;
    const D ph = times(conj(s), 1.0 / r);  // makes S_ik real
    for (int l = threadIdx.x; l < 2 * p; l += kThreads) {  // columns of S, of X
      D* m = l < p ? S + l : X + (l - p);
      const D u = m[i * ld], v = mul(m[k * ld], ph);
      m[i * ld] = axpy(times(u, c), -sn, v);
      m[k * ld] = axpy(times(v, c), sn, u);
    }
    __syncthreads();
    for (int l = threadIdx.x; l < p; l += kThreads) {  // rows of S
      D* m = S + l * ld;
      const D u = m[i], v = mul(m[k], conj(ph));
      m[i] = axpy(times(u, c), -sn, v);
      m[k] = axpy(times(v, c), sn, u);
    }
    __syncthreads();
  }
}

// Residue planes and buffers of one refinement, given back when it ends.
template <class T>
struct Work {
  Dev& d;
  T *A = nullptr, *X = nullptr, *M = nullptr, *S = nullptr, *E = nullptr;
  double *norm = nullptr, *lambda = nullptr, *e2 = nullptr;
  typename Elem<T>::Single* F = nullptr;
  Report* rep = nullptr;
  int* perm = nullptr;
  RnsBlock a, x, y;
  explicit Work(Dev& dev) : d(dev) {}
  ~Work() {
    rns_release(d, a);
    rns_release(d, x);
    rns_release(d, y);
    for (void* q : {static_cast<void*>(A), static_cast<void*>(X), static_cast<void*>(M),
                    static_cast<void*>(S), static_cast<void*>(E), static_cast<void*>(norm),
                    static_cast<void*>(F), static_cast<void*>(rep), static_cast<void*>(perm)})
      if (q) d.release(q);
  }
};

template <class T>
int refine(Dev& d, T* G, int64_t ldg, int p, double* w_dev, bool* done) {
  using D = typename Elem<T>::D;
  using F = typename Elem<T>::F;
  const int64_t ld = p;
  const size_t n = static_cast<size_t>(p) * p;
  Work<T> w(d);
  CHASE_TRY(d.alloc(&w.A, n));
  CHASE_TRY(d.alloc(&w.X, n));
  CHASE_TRY(d.alloc(&w.M, n));
  CHASE_TRY(d.alloc(&w.S, n));
  CHASE_TRY(d.alloc(&w.E, n));
  CHASE_TRY(d.alloc(&w.norm, 3 * static_cast<size_t>(p)));
  w.lambda = w.norm + p;
  w.e2 = w.lambda + p;
  CHASE_TRY(d.alloc(&w.rep, 1));
  CHASE_TRY(d.alloc(&w.perm, static_cast<size_t>(p)));
  auto dp = [](T* q) { return reinterpret_cast<D*>(q); };
  CHASE_CUDA(cudaMemsetAsync(w.rep, 0, sizeof(Report), d.st));
  centre_kernel<D><<<p, kThreads, 0, d.st>>>(dp(G), ldg, p, dp(w.A), ld, w.norm, w.rep);
  note_launch();
  if (p <= kJacobiMax) {
    auto launch = [&](auto rows) -> int {
      constexpr int R = decltype(rows)::value;
      auto kernel = jacobi_kernel<R, D, F>;
      static const cudaError_t ready =
          cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               32 * R * 32 * R * static_cast<int>(sizeof(F)));
      CHASE_CUDA(ready);
      kernel<<<1, kJacobiThreads, sizeof(F) * n, d.st>>>(dp(w.A), ld, p, w.norm, dp(w.X), ld);
      note_launch();
      CHASE_CUDA(cudaGetLastError());
      return CHASE_OK;
    };
    CHASE_TRY(p <= 32   ? launch(std::integral_constant<int, 1>())
              : p <= 64 ? launch(std::integral_constant<int, 2>())
                        : launch(std::integral_constant<int, 3>()));
  } else {
    CHASE_TRY(d.alloc(&w.F, n));
    narrow_kernel<D, F><<<p, kThreads, 0, d.st>>>(dp(w.A), ld, p, w.norm,
                                                  reinterpret_cast<F*>(w.F), ld);
    note_launch();
    CHASE_CUDA(cudaGetLastError());
    const int st = eigh_device(d, w.F, ld, p, w.lambda);
    if (st == CHASE_EIGENSOLVER_ERROR) return CHASE_OK;  // not done
    CHASE_TRY(st);
    CHASE_TRY(launch_convert(d, w.F, ld, w.X, ld, p, p));
  }
  CHASE_TRY(rns_columns(d, w.A, ld, p, p, w.a));
  Report rep;
  std::vector<double> lam(2 * static_cast<size_t>(p));  // eigenvalues, squared column norms of E
  for (int it = 0; it < 8; ++it) {
    CHASE_TRY(rns_columns(d, w.X, ld, p, p, w.x));
    CHASE_TRY(rns_dense(d, w.x, true, w.x, w.M, ld, 1.0, 0.0));
    CHASE_TRY(rns_dense(d, w.a, true, w.x, w.E, ld, 1.0, 0.0));  // A X (A is Hermitian)
    CHASE_TRY(rns_columns(d, w.E, ld, p, p, w.y));
    CHASE_TRY(rns_dense(d, w.x, true, w.y, w.S, ld, 1.0, 0.0));
    rns_release(d, w.x);
    rns_release(d, w.y);
    CHASE_CUDA(cudaMemsetAsync(&w.rep->npairs, 0, sizeof(int), d.st));
    correction_kernel<D><<<p, kThreads, sizeof(double) * p, d.st>>>(
        dp(w.S), dp(w.M), ld, p, w.norm, dp(w.E), w.lambda, w.e2, w.rep);
    note_launch();
    CHASE_CUDA(cudaGetLastError());
    CHASE_CUDA(cudaMemcpyAsync(&rep, w.rep, sizeof(rep), cudaMemcpyDeviceToHost, d.st));
    CHASE_CUDA(cudaMemcpyAsync(lam.data(), w.lambda, sizeof(double) * lam.size(),
                               cudaMemcpyDeviceToHost, d.st));
    CHASE_TRY(d.sync_check("projected eigenproblem"));
    if (rep.npairs > kMaxPairs) return CHASE_OK;
    if (rep.npairs > 0) {
      Pairs pr{};
      pr.n = rep.npairs;
      std::vector<std::pair<int, int>> v;
      for (int k = 0; k < pr.n; ++k) v.emplace_back(rep.pair[k][0], rep.pair[k][1]);
      std::sort(v.begin(), v.end());  // the order does not depend on the blocks'
      for (int k = 0; k < pr.n; ++k) {
        pr.pair[k][0] = v[k].first;
        pr.pair[k][1] = v[k].second;
      }
      rotate_kernel<D><<<1, kThreads, 0, d.st>>>(dp(w.S), dp(w.X), ld, p, pr);
      note_launch();
      CHASE_CUDA(cudaGetLastError());
      continue;
    }
    double e2 = 0.0;
    for (int j = 0; j < p; ++j) e2 += lam[p + j];
    if (!(e2 <= 0.01 * p)) return CHASE_OK;  // nowhere near, or not finite
    CHASE_TRY(rns_rows(d, w.X, ld, p, p, w.x));
    CHASE_TRY(rns_columns(d, w.E, ld, p, p, w.y));
    CHASE_TRY(rns_dense(d, w.x, false, w.y, w.X, ld, 1.0, 1.0));
    rns_release(d, w.x);
    rns_release(d, w.y);
    if (e2 > 1e-16) continue;
    // ascending order (close pairs may have changed places)
    std::vector<int> perm(p);
    std::iota(perm.begin(), perm.end(), 0);
    std::stable_sort(perm.begin(), perm.end(), [&](int i, int j) { return lam[i] < lam[j]; });
    std::vector<double> out(p);
    for (int j = 0; j < p; ++j) out[j] = lam[perm[j]] + rep.centre;
    CHASE_CUDA(cudaMemcpyAsync(w.perm, perm.data(), sizeof(int) * p, cudaMemcpyHostToDevice, d.st));
    CHASE_CUDA(cudaMemcpyAsync(w_dev, out.data(), sizeof(double) * p, cudaMemcpyHostToDevice, d.st));
    CHASE_TRY(launch_permute_cols(d, w.X, ld, G, ldg, p, p, w.perm, false));
    *done = true;
    return d.sync_check("projected eigenproblem");  // the host arrays end here
  }
  return CHASE_OK;
}

// From this size on the refined FP32 solve is the faster one; up to there its
// eigenvalues fit the shared memory of correction_kernel.
constexpr int kRefineMin = 8, kRefineMax = 4096;

template <class T>
int eigh_fp64(Dev& d, T* G, int64_t ldg, int p, double* w_dev) {
  if (p >= kRefineMin && p <= kRefineMax) {
    bool done = false;
    const int st = refine(d, G, ldg, p, w_dev, &done);
    if (st != CHASE_OK && st != CHASE_OUT_OF_MEMORY) return st;
    if (done) return CHASE_OK;
  }
  return eigh_device(d, G, ldg, p, w_dev);
}
}  // namespace

int eigh(Dev& d, chase_c64* G, int64_t ldg, int p, double* w_dev) {
  return eigh_fp64(d, G, ldg, p, w_dev);
}
int eigh(Dev& d, double* G, int64_t ldg, int p, double* w_dev) {
  return eigh_fp64(d, G, ldg, p, w_dev);
}
int eigh(Dev& d, chase_c32* G, int64_t ldg, int p, double* w_dev) {
  return eigh_device(d, G, ldg, p, w_dev);
}
int eigh(Dev& d, float* G, int64_t ldg, int p, double* w_dev) {
  return eigh_device(d, G, ldg, p, w_dev);
}

}  // namespace chase
