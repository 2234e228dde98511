// cqr_adjoint.cu -- kernels of the reverse-mode (adjoint) pass through the coded QR and the
// least-squares solve.
//
// QR adjoint (the coded method's outputs Q = G_0 Q_1, R with G_0 A = Q R, Q^T Q = I): for a
// loss with gradients Qbar, Rbar,
//   M = R Rbar^T - Qbar^T Q,   Bbar = (Qbar + Q copyltu(M)) R^{-T},   Abar = G_0^T Bbar,
// copyltu(M) = tril(M) + tril(M, -1)^T.  This is the standard reverse rule of a thin QR with
// positive diagonal (e.g. Walter & Lehmann 2018, Seeger et al. 2017) applied to G_0 A,
// followed by the chain rule through the linear map A -> G_0 A.
// Least-squares adjoint (x = argmin |A x - y|, A of full column rank): with g = xbar,
//   z = (A^T A)^{-1} g,   r = y - A x,   Abar = r z^T - (A z) x^T,   ybar = A z,
// where A^T A = R^T (Q_1^T Q_1) R and Q_1^T Q_1 = I - Q_2^T Q_2 (coded factors), so
// z = R^{-1} (I - Q_2^T Q_2)^{-1} R^{-T} g.
//
// The building blocks here: a tiled FP32/FP64 GEMM with transposes, copyltu, and a
// triangular solve from the right, X op(R) = B, row blocks in shared memory.
#include <math.h>

#include <algorithm>

#include "cqr_device.cuh"
#include "cqr_kernels.cuh"

namespace cqr {

namespace {

constexpr int kGT = 64;  // GEMM tile (rows and columns of C)
constexpr int kGK = 16;  // GEMM K step

// C (M x N) = alpha op(A) op(B) + beta C; op(A) M x K, op(B) K x N; column-major operands.
// 256 threads; thread (tx, ty) owns rows ty + 16 a and columns tx + 16 b (a, b < 4) of the tile.
template <typename T>
__global__ void __launch_bounds__(256) k_gemm(int ta, int tb, int64_t M, int64_t N, int64_t K,
                                              T alpha, const T* __restrict__ A, int64_t lda,
                                              const T* __restrict__ B, int64_t ldb, T beta,
                                              T* __restrict__ C, int64_t ldc) {
  __shared__ T As[kGK][kGT + 1];  // As[k][i] = op(A)[i0 + i][k0 + k]
  __shared__ T Bs[kGK][kGT + 1];  // Bs[k][j] = op(B)[k0 + k][j0 + j]
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  const int64_t i0 = (int64_t)blockIdx.x * kGT, j0 = (int64_t)blockIdx.y * kGT;
  T acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = T(0);
  for (int64_t k0 = 0; k0 < K; k0 += kGK) {
    for (int e = tid; e < kGT * kGK; e += 256) {
      // consecutive threads walk the contiguous index of the stored operand
      int i, k;
      if (!ta) { i = e % kGT; k = e / kGT; } else { k = e % kGK; i = e / kGK; }
      const int64_t gi = i0 + i, gk = k0 + k;
      T v = T(0);
      if (gi < M && gk < K) v = ta ? A[gk + gi * lda] : A[gi + gk * lda];
      As[k][i] = v;
      int j;
      if (!tb) { k = e % kGK; j = e / kGK; } else { j = e % kGT; k = e / kGT; }
      const int64_t gj = j0 + j, gk2 = k0 + k;
      T w = T(0);
      if (gj < N && gk2 < K) w = tb ? B[gj + gk2 * ldb] : B[gk2 + gj * ldb];
      Bs[k][j] = w;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kGK; ++k) {
      T av[4], bv[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) av[a] = As[k][ty + 16 * a];
#pragma unroll
      for (int b = 0; b < 4; ++b) bv[b] = Bs[k][tx + 16 * b];
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] += av[a] * bv[b];
    }
    __syncthreads();
  }
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int64_t gi = i0 + ty + 16 * a, gj = j0 + tx + 16 * b;
      if (gi < M && gj < N) {
        T* cp = C + gi + gj * ldc;
        *cp = alpha * acc[a][b] + (beta == T(0) ? T(0) : beta * *cp);
      }
    }
}

// S = copyltu(M): S[i][j] = M[i][j] for i >= j, M[j][i] for i < j (n x n, ld n for both).
template <typename T>
__global__ void k_copyltu(const T* __restrict__ Mm, int64_t n, T* __restrict__ S) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n * n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e % n, j = e / n;
    S[e] = i >= j ? Mm[i + j * n] : Mm[j + i * n];
  }
}

// Y (rows x cols, strides rs / cs) += alpha X (same shape, strides xrs / xcs).
template <typename T>
__global__ void k_axpy2d(int64_t rows, int64_t cols, T alpha, const T* __restrict__ X, int64_t xrs,
                         int64_t xcs, T* __restrict__ Y, int64_t yrs, int64_t ycs, int overwrite) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < rows * cols;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e % rows, j = e / rows;
    T* y = Y + i * yrs + j * ycs;
    const T v = alpha * X[i * xrs + j * xcs];
    *y = overwrite ? v : *y + v;
  }
}

// X R^T = B in place (X overwrites B), R upper triangular n x n (ld ldr), B m x n column-major
// (ld cs): columns solved from the last
// (X[:, j] = (B[:, j] - sum_{k>j} X[:, k] R[j, k]) / R[j, j]).
// One CTA per block of rb <= 32 rows, held in shared memory [rb][n + 1]; right-looking: once
// column j is final, its contribution leaves every column still to be solved.  Thread t works
// on row t % 32 and the columns congruent to t / 32 modulo 8 (all lanes of a warp read the
// same coefficient of R).  Used for diagonal blocks and for a few right-hand sides.
template <typename T>
__global__ void __launch_bounds__(256) k_trsm_right(const T* __restrict__ R, int64_t ldr,
                                                    int n, T* __restrict__ B, int64_t cs,
                                                    int64_t m, int rb) {
  extern __shared__ __align__(16) unsigned char trsm_raw[];
  T* X = reinterpret_cast<T*>(trsm_raw);  // [rb][n + 1]
  const int tid = threadIdx.x, ld = n + 1;
  const int64_t r0 = (int64_t)blockIdx.x * rb;
  const int nrow = (int)((m - r0) < rb ? (m - r0) : rb);
  for (int e = tid; e < nrow * n; e += 256) {
    const int j = e / nrow, r = e % nrow;
    X[r * ld + j] = B[r0 + r + (int64_t)j * cs];
  }
  __syncthreads();
  const int r = tid & 31, grp = tid >> 5;
  for (int j = n - 1; j >= 0; --j) {
    if (tid < nrow) X[tid * ld + j] /= R[j + (int64_t)j * ldr];
    __syncthreads();
    if (r < nrow) {
      const T xj = X[r * ld + j];
      for (int k = grp; k < j; k += 8) X[r * ld + k] -= xj * R[k + (int64_t)j * ldr];
    }
    __syncthreads();
  }
  for (int e = tid; e < nrow * n; e += 256) {
    const int j = e / nrow, r2 = e % nrow;
    B[r0 + r2 + (int64_t)j * cs] = X[r2 * ld + j];
  }
}

// R^T x = b in place for R upper triangular (n x n), one CTA per right-hand side (x + blockIdx.x
// ldx): blocks of 64, the diagonal block staged in shared memory and solved by one warp, then every
// later entry less its column's product with the solved block (a warp per eight columns, lanes
// on rows).  Bound by that chain; the blocked right solve took 80 us per block (n = 1024: 1.3 ms).
constexpr int kVT = 1024;
template <typename T>
__global__ void __launch_bounds__(kVT) k_trsv_upper_t(const T* __restrict__ R, int64_t ldr, int64_t n,
                                                      T* __restrict__ x, int64_t ldx) {
  CQR_CHECK(ldr >= n && ldx >= n, 801);
  __shared__ T D[64][65], xs[64];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  T* b = x + (int64_t)blockIdx.x * ldx;
  for (int64_t j0 = 0; j0 < n; j0 += 64) {
    const int jb = (int)(n - j0 < 64 ? n - j0 : 64);
    for (int e = tid; e < 64 * jb; e += kVT) {
      const int i = e & 63, k = e >> 6;
      D[i][k] = i <= k ? R[j0 + i + (j0 + k) * ldr] : T(0);
    }
    __syncthreads();
    if (warp == 0) {
      T v0 = lane < jb ? b[j0 + lane] : T(0), v1 = lane + 32 < jb ? b[j0 + lane + 32] : T(0);
      const T i0 = lane < jb ? T(1) / D[lane][lane] : T(0);
      const T i1 = lane + 32 < jb ? T(1) / D[lane + 32][lane + 32] : T(0);
      for (int j = 0; j < jb; ++j) {
        const T xj = __shfl_sync(0xffffffffu, j < 32 ? v0 * i0 : v1 * i1, j & 31);
        if (lane == (j & 31)) {
          if (j < 32) v0 = xj; else v1 = xj;
        }
        if (lane > j && lane < jb) v0 -= D[j][lane] * xj;
        if (lane + 32 > j && lane + 32 < jb) v1 -= D[j][lane + 32] * xj;
      }
      xs[lane] = v0;
      xs[lane + 32] = v1;
      if (lane < jb) b[j0 + lane] = v0;
      if (lane + 32 < jb) b[j0 + lane + 32] = v1;
    }
    __syncthreads();
    const T x0 = xs[lane], x1 = xs[lane + 32];  // zero past jb
    for (int64_t k0 = j0 + 64 + 8 * warp; k0 < n; k0 += 8 * (kVT / 32)) {
      T a[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const T* r = R + j0 + (k0 + u < n ? k0 + u : n - 1) * ldr;
        a[u] = r[lane] * x0 + r[lane + 32] * x1;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int u = 0; u < 8; ++u) a[u] += __shfl_xor_sync(0xffffffffu, a[u], o);
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (lane == u && k0 + u < n) b[k0 + u] -= a[u];
    }
    __syncthreads();
  }
}

// y = alpha A x + beta y for a few columns (grid.y): 32 rows per CTA, lanes on rows, the eight
// warps on interleaved columns of A; reads A once per column (8192 x 1024: 176 us as a 64 x 64
// tiled product of one column before).
template <typename T>
__global__ void __launch_bounds__(256) k_gemv_n(int64_t M, int64_t K, T alpha, const T* __restrict__ A,
                                                int64_t lda, const T* __restrict__ X, int64_t ldx,
                                                T beta, T* __restrict__ Y, int64_t ldy) {
  CQR_CHECK(lda >= M && ldx >= K && ldy >= M, 802);
  __shared__ T s[8][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t i = (int64_t)blockIdx.x * 32 + lane;
  const T* x = X + (int64_t)blockIdx.y * ldx;
  const T* a = A + (i < M ? i : M - 1);
  T acc[4] = {T(0), T(0), T(0), T(0)};
  int64_t k = warp;
  for (; k + 24 < K; k += 32)
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[u] += a[(k + 8 * u) * lda] * x[k + 8 * u];
  for (; k < K; k += 8) acc[0] += a[k * lda] * x[k];
  s[warp][lane] = (acc[0] + acc[1]) + (acc[2] + acc[3]);
  __syncthreads();
  if (warp == 0 && i < M) {
    T t = T(0);
#pragma unroll
    for (int w = 0; w < 8; ++w) t += s[w][lane];
    T* y = Y + i + (int64_t)blockIdx.y * ldy;
    *y = alpha * t + (beta == T(0) ? T(0) : beta * *y);
  }
}

// C (M x N) += A B^T - D E^T for k columns of A, D (M x k) and B, E (N x k): one pass over C.
template <typename T>
__global__ void __launch_bounds__(256) k_rank2(int64_t M, int64_t N, int k, const T* __restrict__ A,
                                               int64_t lda, const T* __restrict__ B, int64_t ldb,
                                               const T* __restrict__ D, int64_t ldd,
                                               const T* __restrict__ E, int64_t lde,
                                               T* __restrict__ C, int64_t ldc) {
  CQR_CHECK(lda >= M && ldd >= M && ldb >= N && lde >= N && ldc >= M, 803);
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= M) return;
  const int64_t j0 = (int64_t)blockIdx.y * 16;
#pragma unroll 4
  for (int64_t j = j0; j < (j0 + 16 < N ? j0 + 16 : N); ++j) {
    T s = T(0);
    for (int q = 0; q < k; ++q)
      s += A[i + q * lda] * B[j + q * ldb] - D[i + q * ldd] * E[j + q * lde];
    C[i + j * ldc] += s;
  }
}

// Inverses of the kIB x kIB diagonal blocks of R (upper triangular, n x n), one CTA each, into
// V + block * kIB * kIB (column-major, ld kIB, zero below the diagonal): column c of a block by
// thread c, back substitution.
constexpr int kIB = 128;
template <typename T>
__global__ void __launch_bounds__(kIB) k_tri_inverse(const T* __restrict__ R, int64_t ldr, int64_t n,
                                                     T* __restrict__ V) {
  CQR_CHECK(ldr >= n, 804);
  extern __shared__ __align__(16) unsigned char inv_raw[];
  T* U = reinterpret_cast<T*>(inv_raw);  // [kIB][kIB + 1] rows of the block
  T* X = U + kIB * (kIB + 1);            // [kIB][kIB + 1]
  const int64_t j0 = (int64_t)blockIdx.x * kIB;
  const int nb = (int)(n - j0 < kIB ? n - j0 : kIB), c = threadIdx.x;
  for (int e = c; e < nb * kIB; e += kIB) {
    const int i = e % kIB, k = e / kIB;
    if (i < nb) U[i * (kIB + 1) + k] = i <= k ? R[j0 + i + (j0 + k) * ldr] : T(0);
  }
  __syncthreads();
  if (c < nb) {
    for (int k = c; k >= 0; --k) {
      const T* u = U + k * (kIB + 1);
      T s0 = k == c ? T(1) : T(0), s1 = T(0), s2 = T(0), s3 = T(0);
      int i = k + 1;
      for (; i + 3 <= c; i += 4) {
        s0 -= u[i] * X[i * (kIB + 1) + c];
        s1 -= u[i + 1] * X[(i + 1) * (kIB + 1) + c];
        s2 -= u[i + 2] * X[(i + 2) * (kIB + 1) + c];
        s3 -= u[i + 3] * X[(i + 3) * (kIB + 1) + c];
      }
      for (; i <= c; ++i) s0 -= u[i] * X[i * (kIB + 1) + c];
      X[k * (kIB + 1) + c] = ((s0 + s1) + (s2 + s3)) / u[k];
    }
  }
  T* v = V + (int64_t)blockIdx.x * kIB * kIB + (int64_t)c * kIB;
  for (int k = 0; k < kIB; ++k) v[k] = (c < nb && k <= c) ? X[k * (kIB + 1) + c] : T(0);
}

template <typename T>
cudaError_t trsm_unblocked(const T* R, int64_t ldr, int n, T* B, int64_t cs, int64_t m,
                           cudaStream_t st) {
  const size_t cap = 200 * 1024;
  int rb = (int)std::min<int64_t>(32, (int64_t)(cap / ((size_t)(n + 1) * sizeof(T))));
  if (rb < 1) return cudaErrorInvalidValue;  // n too large for one row in shared memory
  const size_t smem = (size_t)rb * (n + 1) * sizeof(T);
  cudaError_t e = cudaFuncSetAttribute(k_trsm_right<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  const unsigned grid = (unsigned)((m + rb - 1) / rb);
  k_trsm_right<T><<<grid, 256, smem, st>>>(R, ldr, n, B, cs, m, rb);
  return cudaGetLastError();
}

}  // namespace

template <typename T>
cudaError_t launch_gemm_general(int ta, int tb, int64_t M, int64_t N, int64_t K, T alpha,
                                const T* A, int64_t lda, const T* B, int64_t ldb, T beta, T* C,
                                int64_t ldc, cudaStream_t st) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  // a few columns: by columns, where the tile of 64 would be nearly empty
  if (!ta && !tb && N <= 8 && K > 0) {
    k_gemv_n<T><<<dim3((unsigned)((M + 31) / 32), (unsigned)N), 256, 0, st>>>(M, K, alpha, A, lda, B,
                                                                             ldb, beta, C, ldc);
    return cudaGetLastError();
  }
  const dim3 grid((unsigned)((M + kGT - 1) / kGT), (unsigned)((N + kGT - 1) / kGT));
  k_gemm<T><<<grid, 256, 0, st>>>(ta, tb, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_copyltu(const T* Mm, int64_t n, T* S, cudaStream_t st) {
  const int blocks = (int)std::min<int64_t>(1024, (n * n + 255) / 256);
  k_copyltu<T><<<blocks, 256, 0, st>>>(Mm, n, S);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_axpy2d(int64_t rows, int64_t cols, T alpha, const T* X, int64_t xrs, int64_t xcs,
                          T* Y, int64_t yrs, int64_t ycs, bool overwrite, cudaStream_t st) {
  if (rows <= 0 || cols <= 0) return cudaSuccess;
  const int blocks = (int)std::min<int64_t>(2048, (rows * cols + 255) / 256);
  k_axpy2d<T><<<blocks, 256, 0, st>>>(rows, cols, alpha, X, xrs, xcs, Y, yrs, ycs, overwrite ? 1 : 0);
  return cudaGetLastError();
}

// Blocked: diagonal blocks of kTB columns, from the last, are solved by the row-block kernel, the
// rest of each step is one GEMM update, B[:, K] -= X[:, J] R[K, J]^T for the blocks K < J.
template <typename T>
cudaError_t launch_trsm_right(const T* R, int64_t ldr, int64_t n, T* B, int64_t cs, int64_t m,
                              cudaStream_t st) {
  if (m <= 0 || n <= 0) return cudaSuccess;
  constexpr int kTB = 64;
  for (int64_t J = (n + kTB - 1) / kTB - 1; J >= 0; --J) {
    const int64_t j0 = J * kTB, jb = std::min<int64_t>(kTB, n - j0);
    cudaError_t e = trsm_unblocked<T>(R + j0 + j0 * ldr, ldr, (int)jb, B + j0 * cs, cs, m, st);
    if (e == cudaSuccess && j0 > 0)
      e = launch_gemm_general<T>(0, 1, m, j0, jb, T(-1), B + j0 * cs, cs, R + j0 * ldr, ldr, T(1), B, cs,
                                 st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// R^T x = b in place, k right-hand sides.
template <typename T>
cudaError_t launch_trsv_upper_t(const T* R, int64_t ldr, int64_t n, T* x, int64_t ldx, int64_t k,
                                cudaStream_t st) {
  if (n <= 0 || k <= 0) return cudaSuccess;
  k_trsv_upper_t<T><<<(unsigned)k, kVT, 0, st>>>(R, ldr, n, x, ldx);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_rank2(int64_t M, int64_t N, int k, const T* A, int64_t lda, const T* B, int64_t ldb,
                         const T* D, int64_t ldd, const T* E, int64_t lde, T* C, int64_t ldc,
                         cudaStream_t st) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  const dim3 grid((unsigned)((M + 255) / 256), (unsigned)((N + 15) / 16));
  k_rank2<T><<<grid, 256, 0, st>>>(M, N, k, A, lda, B, ldb, D, ldd, E, lde, C, ldc);
  return cudaGetLastError();
}

int tri_inverse_block() { return kIB; }

template <typename T>
cudaError_t launch_tri_inverse(const T* R, int64_t ldr, int64_t n, T* V, cudaStream_t st) {
  const size_t smem = (size_t)2 * kIB * (kIB + 1) * sizeof(T);
  cudaError_t e = cudaFuncSetAttribute(k_tri_inverse<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  k_tri_inverse<T><<<(unsigned)((n + kIB - 1) / kIB), kIB, smem, st>>>(R, ldr, n, V);
  return cudaGetLastError();
}
template cudaError_t launch_tri_inverse<float>(const float*, int64_t, int64_t, float*, cudaStream_t);

cudaError_t bounds_take_adjoint(int* code, int* site) { return bounds_take_here(code, site); }

#define CQR_ADJ_INSTANTIATE(T)                                                                   \
  template cudaError_t launch_gemm_general<T>(int, int, int64_t, int64_t, int64_t, T, const T*,  \
                                              int64_t, const T*, int64_t, T, T*, int64_t,        \
                                              cudaStream_t);                                     \
  template cudaError_t launch_copyltu<T>(const T*, int64_t, T*, cudaStream_t);                   \
  template cudaError_t launch_trsv_upper_t<T>(const T*, int64_t, int64_t, T*, int64_t, int64_t,   \
                                              cudaStream_t);                                     \
  template cudaError_t launch_rank2<T>(int64_t, int64_t, int, const T*, int64_t, const T*, int64_t, \
                                       const T*, int64_t, const T*, int64_t, T*, int64_t,        \
                                       cudaStream_t);                                            \
  template cudaError_t launch_axpy2d<T>(int64_t, int64_t, T, const T*, int64_t, int64_t, T*,     \
                                        int64_t, int64_t, bool, cudaStream_t);                   \
  template cudaError_t launch_trsm_right<T>(const T*, int64_t, int64_t, T*, int64_t, int64_t,    \
                                            cudaStream_t);

CQR_ADJ_INSTANTIATE(float)
CQR_ADJ_INSTANTIATE(double)

}  // namespace cqr
