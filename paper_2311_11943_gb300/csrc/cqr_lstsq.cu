// cqr_lstsq.cu -- the middle factor of the tall least squares (a9) and of its adjoint:
// (I - Q_2^T Q_2) w = z, z = Q_1^T y (or given), I - Q_2^T Q_2 = Q_1^T Q_1 by the orthonormality of
// the coded Q.  SPD with condition number at most 1 + ||G~||^2, a property of the code.
//
// Iterative refinement: the residual r = z - w + Q_2^T (Q_2 w) and w in FP64, the corrections by
// conjugate gradients in FP32 to five or six digits, until |r| <= 1e-15 |z| (the accuracy of
// conjugate gradients in FP64 throughout; 1e-11 where the result is FP32, see Ends) or no longer
// falling.  Two to four FP64 residuals instead of some ninety FP64 iterations: the FP64 pipes give about two products per cycle and SM, the
// FP32 ones 128, and an iteration is then one pass over Q_2 and one sum over the CTAs.
// G CTAs each hold rows of Q_2 in shared memory (transposed while they are loaded, so that both
// products read along rows), every vector of n entries is held by every CTA, and the n sums of
// Q_2^T t go through cqr_exchange.cuh: one exchange per iteration instead of four grid
// barriers, and no traffic for Q_2.  Measured, FP64 iterations on 32 CTAs before, this after
// (FP32, one right-hand side): Q_2 2048 x 2048 12.3 and 0.73 ms, 1538 x 1320 3.5 and 0.36 ms.
#include <math.h>

#include <algorithm>

#include "cqr_exchange.cuh"
#include "cqr_kernels.cuh"

namespace cqr {

namespace {

constexpr int kNT = 512;
constexpr int kNW = kNT / 32;
constexpr size_t kSmemCap = 227 * 1024;
constexpr int kMaxRhs = 4;  // right-hand sides of one launch
constexpr int kMaxOuter = 12, kMaxInner = 80;
// Ends, as squares: of the refinement (|r| over |z|) and of one correction (over its |r|).  With
// FP64 results 1e-15 and three or four corrections of 1e-5; with FP32 results 1e-11, where the
// error of w is at most the condition number times that, a hundredth of the rounding of w to FP32
// for a condition number of 60, and two corrections of 1.7e-6 reach it.
template <typename T>
struct Ends {
  static constexpr double kOuter = sizeof(T) == 8 ? 1e-30 : 1e-22;
  static constexpr float kInner = sizeof(T) == 8 ? 1e-10f : 3e-12f;
};
constexpr unsigned kTags = kMaxOuter * (kMaxInner + 1) + 8;
// CTAs for e entries of Q_2: one per kFew entries up to kGroup CTAs (an exchange costs about
// 2 us, a CTA's pass over 32,000 entries 3.7), then no more until each has kMany (problems on
// other streams want SMs too).
constexpr int64_t kFew = 4096, kMany = 24000, kGroup = 43;

// (double)f by integer operations where f is a normal number: a conversion takes the FP64 pipe.
__device__ __forceinline__ double widen(float f) {
  const int b = __float_as_int(f);
  const int ex = b & 0x7f800000;
  if (ex == 0 || ex == 0x7f800000) return (double)f;
  return __hiloint2double((b & 0x80000000) | (((b & 0x7fffffff) >> 3) + 0x38000000), b << 29);
}
__device__ __forceinline__ double widen(double f) { return f; }
struct alignas(16) F4 { float v[4]; };
struct alignas(16) D2 { double v[2]; };
__device__ __forceinline__ void ld4(const float* p, float* x) {
  const F4 a = *reinterpret_cast<const F4*>(p);
#pragma unroll
  for (int u = 0; u < 4; ++u) x[u] = a.v[u];
}
__device__ __forceinline__ void ld4(const double* p, double* x) {
  const D2 a = *reinterpret_cast<const D2*>(p), b = *reinterpret_cast<const D2*>(p + 2);
  x[0] = a.v[0]; x[1] = a.v[1]; x[2] = b.v[0]; x[3] = b.v[1];
}
template <typename R, typename T>
__device__ __forceinline__ R as(T x) {
  if constexpr (sizeof(R) == 8) return widen(x);
  else return (float)x;
}

// z = Q_1^T y in FP64, a warp per column, a row of the grid per right-hand side; z = u when u is
// given.
template <typename T>
__global__ void __launch_bounds__(256) k_ls_rhs(const T* __restrict__ Q, int64_t ldq, int64_t m,
                                                int64_t n, const T* __restrict__ y, int64_t ldy,
                                                const T* __restrict__ u, int64_t ldu,
                                                double* __restrict__ z) {
  CQR_CHECK(ldq >= m, 601);
  z += (int64_t)blockIdx.y * n;
  y += (int64_t)blockIdx.y * ldy;
  const int lane = threadIdx.x & 31;
  const int64_t j = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (j >= n) return;
  if (u) {
    if (lane == 0) z[j] = (double)u[(int64_t)blockIdx.y * ldu + j];
    return;
  }
  const T* q = Q + j * ldq;
  double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
  int64_t i = lane;
  for (; i + 96 < m; i += 128) {
    const T q0 = q[i], q1 = q[i + 32], q2 = q[i + 64], q3 = q[i + 96];
    const T y0 = y[i], y1 = y[i + 32], y2 = y[i + 64], y3 = y[i + 96];
    a0 = fma(widen(q0), widen(y0), a0);
    a1 = fma(widen(q1), widen(y1), a1);
    a2 = fma(widen(q2), widen(y2), a2);
    a3 = fma(widen(q3), widen(y3), a3);
  }
  for (; i < m; i += 32) a0 = fma(widen(q[i]), widen(y[i]), a0);
  const double s = warp_sum((a0 + a1) + (a2 + a3));
  if (lane == 0) z[j] = s;
}

struct LsPlan {
  int G, rb;      // CTAs, rows of Q_2 per CTA
  int ns;         // padded vector length (a multiple of 128)
  int in_smem;    // the rows are in shared memory (else read from global memory, rb a multiple of 32)
  size_t smem;
};

// Shared memory besides the rows of Q_2.
size_t ls_vec_bytes(int ns, int rb) { return (size_t)ns * 28 + (size_t)(rb + 1) * 8 + kNT * 8 + 64 * 8; }

bool plan_ls(int64_t c, int64_t n, size_t elem, int num_sms, LsPlan* p) {
  if (n > 16384 || c < 1) return false;
  p->ns = (int)((n + 127) / 128 * 128);
  auto fits = [&](int64_t rb) {
    return ls_vec_bytes(p->ns, (int)rb) + (size_t)rb * p->ns * elem + 2048 <= kSmemCap;
  };
  const int64_t e = c * n;
  int64_t G = std::max(std::min((e + kFew - 1) / kFew, kGroup), (e + kMany - 1) / kMany);
  G = std::min<int64_t>(G, num_sms);
  for (; G <= num_sms; G = G < num_sms ? std::min<int64_t>(num_sms, 2 * G) : num_sms + 1) {
    const int64_t rb = (c + G - 1) / G;
    if (!fits(rb)) continue;
    p->rb = (int)rb;
    p->G = (int)((c + rb - 1) / rb);
    p->in_smem = 1;
    p->smem = ls_vec_bytes(p->ns, p->rb) + (size_t)rb * p->ns * elem;
    return true;
  }
  const int64_t rb = 32 * ((c + 32LL * num_sms - 1) / (32LL * num_sms));
  if (ls_vec_bytes(p->ns, (int)rb) + kNW * 33 * 8 + 2048 > kSmemCap) return false;
  p->rb = (int)rb;
  p->G = (int)((c + rb - 1) / rb);
  p->in_smem = 0;
  p->smem = ls_vec_bytes(p->ns, p->rb) + kNW * 33 * 8;
  return true;
}

template <typename R>
__device__ __forceinline__ R block_sum(R v, double* scratch) {
  R* s = reinterpret_cast<R*>(scratch);
  v = warp_sum(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = v;
  __syncthreads();
  R t = R(0);
#pragma unroll
  for (int k = 0; k < kNW; ++k) t += s[k];
  return t;
}

// out[j] = (Q_2^T Q_2 v)_j, this CTA's rows of Q_2, in precision R (products and sums).
template <typename R, typename T>
__device__ __forceinline__ void gram_vec(const T* __restrict__ S, const T* __restrict__ Q2, int64_t ldq,
                                         int rows, int ns, int n, bool in_smem, const R* v, R* t,
                                         R* tp, R* out) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (in_smem) {
    // t = S v: four rows per warp at a time (their sums over the lanes overlap)
    for (int i0 = 4 * warp; i0 < rows; i0 += 4 * kNW) {
      const T* s[4];
      R a[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        s[u] = S + (size_t)min(i0 + u, rows - 1) * ns;
        a[u] = R(0);
      }
      for (int j = 4 * lane; j < ns; j += 128) {  // the padding of v and S is zero
        R vv[4];
        ld4(v + j, vv);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          T q[4];
          ld4(s[u] + j, q);
          a[u] += (as<R>(q[0]) * vv[0] + as<R>(q[1]) * vv[1]) + (as<R>(q[2]) * vv[2] + as<R>(q[3]) * vv[3]);
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int u = 0; u < 4; ++u) a[u] += __shfl_xor_sync(0xffffffffu, a[u], o);
      if (lane < 4 && i0 + lane < rows) t[i0 + lane] = lane == 0 ? a[0] : lane == 1 ? a[1] : lane == 2 ? a[2] : a[3];
    }
    __syncthreads();
    // out = S^T t: a thread per column, or, for few columns, groups of threads on every ng-th row
    const int nw = (n + 31) / 32 * 32, ng = max(1, kNT / nw);
    for (int j0 = 0; j0 < n; j0 += kNT) {
      const int j = ng > 1 ? tid % nw : j0 + tid, grp = ng > 1 ? tid / nw : 0;
      R a0 = R(0);
      if (j < n && grp < ng) {
        const T* s = S + j;
        R a[4] = {R(0), R(0), R(0), R(0)};
        int i = grp;
#pragma unroll 2
        for (; i + 3 * ng < rows; i += 4 * ng)
#pragma unroll
          for (int u = 0; u < 4; ++u) a[u] += as<R>(s[(size_t)(i + u * ng) * ns]) * t[i + u * ng];
        for (; i < rows; i += ng) a[0] += as<R>(s[(size_t)i * ns]) * t[i];
        a0 = (a[0] + a[1]) + (a[2] + a[3]);
      }
      if (ng > 1) {
        tp[tid] = a0;
        __syncthreads();
        if (grp == 0)
          for (int k = 1; k < ng; ++k) a0 += tp[k * nw + j];
      }
      if (j < n && grp == 0) out[j] = a0;
    }
  } else {
    // lanes on rows, the warps on interleaved columns; then a warp per column
    for (int i0 = 0; i0 < rows; i0 += 32) {
      const bool ok = i0 + lane < rows;
      const T* q = Q2 + i0 + (ok ? lane : 0);
      R a = R(0);
      if (ok)
#pragma unroll 16
        for (int j = warp; j < n; j += kNW) a += as<R>(q[(int64_t)j * ldq]) * v[j];
      tp[warp * 33 + lane] = a;
      __syncthreads();
      if (warp == 0) {
        R s = R(0);
        for (int k = 0; k < kNW; ++k) s += tp[k * 33 + lane];
        if (ok) t[i0 + lane] = s;
      }
      __syncthreads();
    }
    constexpr int C = 8;  // columns of a warp in flight
    for (int j0 = warp; j0 < n; j0 += C * kNW) {
      R a[C];
#pragma unroll
      for (int u = 0; u < C; ++u) a[u] = R(0);
      for (int i = lane; i < rows; i += 32)
#pragma unroll
        for (int u = 0; u < C; ++u)
          a[u] += as<R>(Q2[i + (int64_t)min(j0 + u * kNW, n - 1) * ldq]) * t[i];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int u = 0; u < C; ++u) a[u] += __shfl_xor_sync(0xffffffffu, a[u], o);
      if (lane == 0)
#pragma unroll
        for (int u = 0; u < C; ++u)
          if (j0 + u * kNW < n) out[j0 + u * kNW] = a[u];
    }
  }
}

// Row y of the grid does right-hand side y, with sums and a tag count of its own: an iteration is
// an exchange among few CTAs, which other right-hand sides' need not wait for.  1003 x 96, three
// right-hand sides: 0.35 ms one after the other, 0.12 ms side by side.
template <typename T>
__global__ void __launch_bounds__(kNT, 1) k_ls_refine(const T* __restrict__ Q, int64_t ldq,
                                                       int64_t m_pad, int64_t c64, int64_t n64,
                                                       const double* __restrict__ z, T* __restrict__ x,
                                                       int64_t ldx, int rb, int ns, int in_smem,
                                                       unsigned char* xws, int ecap, int* status,
                                                       long long wait_limit) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int tid = threadIdx.x, g = blockIdx.x, n = (int)n64, c = (int)c64;
  CQR_CHECK(ldq >= m_pad + c64 && ns >= n && (int64_t)gridDim.x * rb >= c64 && 2 * n <= ecap &&
                (in_smem || rb % 32 == 0), 602);
  double* w = reinterpret_cast<double*>(smraw);  // [ns]
  double* W = w + ns;                            // [ns] sums (FP32 ones in the same place)
  double* red = W + ns;                          // [kNT]
  double* bs = red + kNT;                        // [64] block sums
  double* t = bs + 64;                           // [rb]
  float* p = reinterpret_cast<float*>(t + (rb + 1) / 2 * 2);  // [ns], 16-byte aligned as what follows
  float* d = p + ns;                             // [ns]
  float* r = d + ns;                             // [ns]
  unsigned char* rest = reinterpret_cast<unsigned char*>(r + ns);
  T* S = reinterpret_cast<T*>(rest);             // in_smem: [rb][ns]
  double* tp = in_smem ? red : reinterpret_cast<double*>(rest);  // [kNT], or [kNW][33]
  float* Wf = reinterpret_cast<float*>(W);
  z += (int64_t)blockIdx.y * n;
  x += (int64_t)blockIdx.y * ldx;
  unsigned* epoch = reinterpret_cast<unsigned*>(xws + blockIdx.y * (256 / kMaxRhs));
  unsigned long long* fin = reinterpret_cast<unsigned long long*>(xws + 256) +
                            (size_t)blockIdx.y * (gridDim.x + 1) * ecap;
  unsigned long long* part = fin + ecap;
  Xch xc{part, fin, ecap, 0u, status, wait_limit};
  const bool ok0 = exchange_begin(xc, epoch, kTags);
  if (!ok0) {  // an earlier error: no factors to solve with
    if (g == 0)
      for (int j = tid; j < n; j += kNT) x[j] = nan_value<T>();
    return;
  }
  const unsigned first = xc.tag;
  const int i0 = g * rb;
  const int rows = max(0, min(rb, c - i0));
  const T* Q2 = Q + m_pad + i0;
  if (in_smem) {
    for (int idx = tid; idx < rows * ns; idx += kNT) {
      const int j = idx / rows, i = idx - j * rows;
      S[(size_t)i * ns + j] = j < n ? Q2[i + (int64_t)j * ldq] : T(0);
    }
  }
  for (int j = tid; j < ns; j += kNT) {
    w[j] = 0.0;
    p[j] = 0.f;
  }
  __syncthreads();
  bool ok = true, finite = true;
  double zz = 0.0, prev = 0.0, rn = 0.0;
  for (int o = 0; o < kMaxOuter; ++o) {
    // W <- r = z - w + Q_2^T Q_2 w in FP64
    if (o > 0) {
      gram_vec<double, T>(S, Q2, ldq, rows, ns, n, in_smem != 0, w, t, tp, W);
      ok = exchange<double, kNT>(xc, W, n, red);
      if (!ok) break;
    }
    double loc = 0.0;
    for (int j = tid; j < n; j += kNT) {
      const double rj = o > 0 ? z[j] - (w[j] - W[j]) : z[j];
      W[j] = rj;
      loc = fma(rj, rj, loc);
    }
    const double rr64 = block_sum(loc, bs);
    if (o == 0) zz = rr64;
    finite = isfinite(rr64);  // a right-hand side or rows of Q_2 that are not: no x (NaN)
    if (!finite) break;
    if (o > 0 && rr64 > prev) {  // the correction made it worse: without it
      for (int j = tid; j < n; j += kNT) w[j] = fma(-rn, (double)d[j], w[j]);
      break;
    }
    if (!(rr64 > Ends<T>::kOuter * zz) || (o > 0 && !(rr64 < 0.25 * prev))) break;
    prev = rr64;
    rn = sqrt(rr64);
    const double irn = 1.0 / rn;
    for (int j = tid; j < n; j += kNT) {
      const float rj = (float)(W[j] * irn);
      r[j] = rj;
      p[j] = rj;
      d[j] = 0.f;
    }
    __syncthreads();
    // d: the correction over |r| by conjugate gradients in FP32
    float rr = 1.f;
    for (int it = 0; it < kMaxInner && rr > Ends<T>::kInner; ++it) {
      gram_vec<float, T>(S, Q2, ldq, rows, ns, n, in_smem != 0, p, reinterpret_cast<float*>(t),
                         reinterpret_cast<float*>(tp), Wf);
      ok = exchange<float, kNT>(xc, Wf, n, reinterpret_cast<float*>(red));
      if (!ok) break;
      float pl = 0.f;
      for (int j = tid; j < n; j += kNT) {
        const float a = p[j] - Wf[j];
        Wf[j] = a;
        pl = fmaf(p[j], a, pl);
      }
      const float pap = block_sum(pl, bs);
      if (!(pap > 0.f)) break;
      const float alpha = rr / pap;
      float rl = 0.f;
      for (int j = tid; j < n; j += kNT) {
        d[j] = fmaf(alpha, p[j], d[j]);
        const float rj = fmaf(-alpha, Wf[j], r[j]);
        r[j] = rj;
        rl = fmaf(rj, rj, rl);
      }
      const float rr2 = block_sum(rl, bs);
      const float beta = rr2 / rr;
      rr = rr2;
      for (int j = tid; j < n; j += kNT) p[j] = fmaf(beta, p[j], r[j]);
      __syncthreads();
    }
    if (!ok) break;
    for (int j = tid; j < n; j += kNT) w[j] = fma(rn, (double)d[j], w[j]);
    __syncthreads();
  }
  exchange_end(epoch, first, kTags);
  if (ok && g == 0)
    for (int j = tid; j < n; j += kNT) x[j] = finite ? (T)w[j] : nan_value<T>();
}

}  // namespace

// Words for the sums of n doubles over num_sms CTAs, and the tag count.
size_t ls_refine_bytes(int64_t n, int num_sms) {
  if (n > 16384) return 256;
  return 256 + (size_t)(num_sms + 1) * 2 * n * 8;
}

// k right-hand sides, as many at a time as the SMs and the words hold.  z: min(k, 4) n doubles of
// workspace; xws: ls_refine_bytes of device memory, zero before the first launch and kept between
// launches.  False in *taken (nothing launched) when the vectors do not fit.
template <typename T>
cudaError_t launch_ls_refine(const T* Q, int64_t ldq, int64_t m, int64_t m_pad, int64_t c, int64_t n,
                             int k, const T* y, int64_t ldy, const T* u, int64_t ldu, T* x,
                             int64_t ldx, double* z, void* xws, int* status, int num_sms,
                             cudaStream_t st, long long wait_limit, bool* taken) {
  LsPlan p{};
  *taken = plan_ls(c, n, sizeof(T), num_sms, &p);
  if (!*taken) return cudaSuccess;
  const void* fn = (const void*)k_ls_refine<T>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smem);
  if (e != cudaSuccess) return e;
  int ecap = (int)(2 * n);
  unsigned char* xw = static_cast<unsigned char*>(xws);
  long long wl = wait_limit > 0 ? wait_limit : kWaitLimitCycles;
  const double* zc = z;
  // one CTA per SM, and (G + 1) ecap words per right-hand side of the (SMs + 1) ecap there are
  const int at_once = std::max(1, std::min({kMaxRhs, num_sms / p.G, (num_sms + 1) / (p.G + 1)}));
  for (int k0 = 0; k0 < k; k0 += at_once) {
    const int kk = std::min(at_once, k - k0);
    k_ls_rhs<T><<<dim3((unsigned)((n + 7) / 8), kk), 256, 0, st>>>(
        Q, ldq, m, n, y ? y + k0 * ldy : nullptr, ldy, u ? u + k0 * ldu : nullptr, ldu, z);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    T* xk = x + k0 * ldx;
    void* args[] = {(void*)&Q, &ldq, &m_pad, &c, &n, &zc, &xk, &ldx, &p.rb, &p.ns, &p.in_smem, &xw,
                    &ecap, &status, &wl};
    e = cudaLaunchCooperativeKernel(fn, dim3(p.G, kk), dim3(kNT), args, p.smem, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template cudaError_t launch_ls_refine<float>(const float*, int64_t, int64_t, int64_t, int64_t, int64_t,
                                             int, const float*, int64_t, const float*, int64_t, float*,
                                             int64_t, double*, void*, int*, int, cudaStream_t, long long,
                                             bool*);
template cudaError_t launch_ls_refine<double>(const double*, int64_t, int64_t, int64_t, int64_t,
                                              int64_t, int, const double*, int64_t, const double*,
                                              int64_t, double*, int64_t, double*, void*, int*, int,
                                              cudaStream_t, long long, bool*);

cudaError_t bounds_take_lstsq(int* code, int* site) { return bounds_take_here(code, site); }

}  // namespace cqr
