// cqr_panel_blk.cu -- panel factorisation of PBMGS (a3) in sub-blocks of S columns: the
// arithmetic of Algorithm CGS with the ICGS reorthogonalisation (Appendix A), with one reduction
// per S columns instead of one per column.
//
// G CTAs of one cooperative launch own contiguous row slices of the panel, resident in shared
// memory.  For the sub-block of columns j .. j+S-1 (P is the panel with columns < j done):
//   W = P_S^T P[:, j:b]                        one reduction of S (b - j) sums over the CTAs
//   U^T U = W[:, 0:S]                          Cholesky, U = the rows j.. of R in the sub-block
//   R[j:j+S, j+S:b] = U^{-T} W[:, S:]
//   Q_S = P_S U^{-1},  P[:, j+S:b] -= Q_S R[j:j+S, j+S:b]
// which are the same q and r as S steps of the column recurrence.  The pivot u_kk^2 is the
// squared norm v of column j+k after its projections, so the ICGS test v < tau^2 eta is taken on
// it.  When a column of the sub-block fails the test, the sub-block is projected once more on
// all computed columns of the panel before the update (two more reductions per column become
// one per sub-block):
//   T = P_S U^{-1},  Z1 = Q[:, 0:j]^T T,  U2^T U2 = T^T T - Z1^T Z1,  Q_S = (T - Q[:, 0:j] Z1) U2^{-1},
//   R[0:j, S] += Z1 U,  R[j:j+S, j:b] = U2 U and U2^{-T} U^{-T} W[:, S:].
// The Cholesky form and the column recurrence differ by rounding of order u times the squared
// condition number of the sub-block.  Where a row of U^{-T} amplifies rounding by more than
// kMaxAmp (the sum over k of |U^{-T}_ak| |p_k|, 1 for orthogonal columns; nearly dependent columns)
// the sub-block always takes the second projection, and three things change so that no digit
// depends on the first factor: T = P_S U^{-1} by substitution (P_S = T U to rounding), the
// rows of R behind the sub-block from products with T (the second projection's products then
// run over all columns), and a pivot below kFloor times its column's squared norm is raised to
// that, which only scales its column of T.  The sub-block ends before a column with amplification
// above kMaxHard or a pivot that is not positive and finite, and, in the second factor, before
// one of whose norm the projection leaves less than half (its pivot has lost its digits; it is given
// back as T U).  That column goes through the column recurrence itself (products, ICGS
// reorthogonalisation when the test asks for it, normalisation, update), and the next sub-block
// starts behind it.  Without the ICGS test (MGS) the second projection is within the
// sub-block.  Every CTA takes the same decisions from the same sums.
// Why not the recurrence for every column above kMaxAmp: 4096 x 2048, b = 128, every second column
// within 1e-3 of the one before, 24.5 ms that way (8.4 ms by the column-by-column kernels), 4.8 ms
// so; every seventh column 7.7 (5.8), 4.8 ms.
//
// Why: the panel is bound by the latency of its reductions and by passes over the slice.  Per
// column, one exchange and one pass over the slice cost 2.2 us (5120 x 128, one cluster of 16)
// and 4.5 us (20480 x 256, 112 CTAs); per S columns the same two cost a few microseconds,
// the slice is read twice and written once, and every SM can take part.
//
// The reductions are cqr_exchange.cuh's.
#include <math.h>
#include <stdlib.h>

#include <algorithm>

#include "cqr_device.cuh"
#include "cqr_exchange.cuh"
#include "cqr_kernels.cuh"
#include "cqr_subblock.cuh"

namespace cqr {

namespace {

constexpr int kNT = 512;
constexpr int kNW = kNT / 32;
constexpr int kMaxB = 512;            // widest panel
constexpr size_t kSmemCap = 227 * 1024;
// A second projection whose products differ from the identity by less than kNearI needs no
// Cholesky: U = I + E / 2 on the diagonal and I + E above it, with E^2 below rounding.
template <typename T>
constexpr T kNearI = sizeof(T) == 4 ? T(1.0 / 8192) : T(1.0 / (1 << 27));
// Largest amplification that the second projection mends (u kMaxHard^2 is at most 1/4: T stays well
// conditioned), and the floor of a pivot over its column's squared norm (amplification about
// 1 / sqrt(kFloor) then).
template <typename T>
constexpr float kMaxHard = sizeof(T) == 4 ? 2048.f : 16777216.f;
template <typename T>
constexpr T kFloor = sizeof(T) == 4 ? T(1.0 / (1 << 18)) : T(1.0 / (1ll << 44));
// Row stride of the solved coefficients: 16-byte rows
template <typename T>
constexpr int kSY = kS<T> + 16 / (int)sizeof(T);

template <typename T>
__device__ __forceinline__ T round_up_to(double t);
template <>
__device__ __forceinline__ float round_up_to<float>(double t) { return __double2float_ru(t); }
template <>
__device__ __forceinline__ double round_up_to<double>(double t) { return t; }

// A squared norm as m 4^h, 1 <= m < 4 (h = 0 for floats, whose range holds it), and |x| 2^h as a
// float (zero below its range, infinite above): the test of what a sub-block amplifies multiplies
// entries of U^{-T} by column norms, whose product is a pure number also where neither fits a
// float.  By integer operations on the high word, since the FP64 pipe is slow.
__device__ __forceinline__ float norm_of(float v, int& h) {
  h = 0;
  return sqrtf(v);
}
__device__ __forceinline__ float norm_of(double v, int& h) {
  const int hi = __double2hiint(v);
  if (hi < 0x00100000 || hi >= 0x7ff00000) {  // no pivot comes of it
    h = 0;
    return 0.f;
  }
  const int ex = (hi >> 20) - 1023;
  h = ex >> 1;
  return sqrtf(__int_as_float(((127 + (ex & 1)) << 23) | ((hi & 0xfffff) << 3)));
}
__device__ __forceinline__ float scaled_abs(float x, int) { return fabsf(x); }
__device__ __forceinline__ float scaled_abs(double x, int h) {
  const int hi = __double2hiint(x) & 0x7fffffff;
  const int ex = (hi >> 20) - 1023 + 127 + h;
  if (hi < 0x00100000 || ex <= 0) return 0.f;
  return ex >= 255 || hi >= 0x7ff00000 ? __int_as_float(0x7f800000)
                                       : __int_as_float((ex << 23) | ((hi & 0xfffff) << 3));
}

// Lane a < gd: what row a of U^{-T} amplifies (warp 0), the sum over k of |U^{-T}_ak| |p_k|.
template <typename T>
__device__ __forceinline__ float amplification(const T* sLi, const float* sNrm, const int* sExp, int n, int gd) {
  constexpr int S = kS<T>;
  const int lane = threadIdx.x & 31;
  float amp = 0.f;
  if (lane < gd)
#pragma unroll 4
    for (int k = 0; k < S; ++k) {
      const int q = min(k, n - 1);
      amp += scaled_abs(sLi[lane * S + k], sExp[q]) * sNrm[q];
    }
  return amp;
}

// 16 bytes of a column in shared memory and their arithmetic: four floats as two packed f32x2
// pairs, or two doubles.
__device__ __forceinline__ u64 ffma2(u64 a, u64 b, u64 c) {
  u64 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
template <typename T>
struct Vec;
template <>
struct Vec<float> {
  static constexpr int N = 4;
  struct A { u64 v; };                  // accumulator of a product of vectors
  u64 lo, hi;
  __device__ static Vec ld(const float* p) {
    const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(p);
    return Vec{x.x, x.y};
  }
  __device__ static void st(float* p, Vec v) {
    *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(v.lo, v.hi);
  }
  __device__ static A zero() { return A{0ull}; }
  __device__ static void dot(A& a, Vec x, Vec y) {
    a.v = ffma2(x.lo, y.lo, a.v);
    a.v = ffma2(x.hi, y.hi, a.v);
  }
  __device__ static float sum(A a) {
    float x, y;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v));
    return x + y;
  }
  __device__ static Vec zeros() { return Vec{0ull, 0ull}; }
  __device__ static void fma(Vec& d, Vec x, float c) {
    u64 s;
    asm("mov.b64 %0, {%1, %1};" : "=l"(s) : "f"(c));
    d.lo = ffma2(x.lo, s, d.lo);
    d.hi = ffma2(x.hi, s, d.hi);
  }
  // d += sum over the N scalars of y of x[i] y_i
  __device__ static void fmas(Vec& d, const Vec* x, Vec y) {
    float c0, c1, c2, c3;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(c0), "=f"(c1) : "l"(y.lo));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(c2), "=f"(c3) : "l"(y.hi));
    fma(d, x[0], c0);
    fma(d, x[1], c1);
    fma(d, x[2], c2);
    fma(d, x[3], c3);
  }
};
template <>
struct Vec<double> {
  static constexpr int N = 2;
  struct A { double v; };
  double lo, hi;
  __device__ static Vec ld(const double* p) {
    const double2 x = *reinterpret_cast<const double2*>(p);
    return Vec{x.x, x.y};
  }
  __device__ static void st(double* p, Vec v) {
    *reinterpret_cast<double2*>(p) = make_double2(v.lo, v.hi);
  }
  __device__ static A zero() { return A{0.0}; }
  __device__ static void dot(A& a, Vec x, Vec y) { a.v = ::fma(x.hi, y.hi, ::fma(x.lo, y.lo, a.v)); }
  __device__ static double sum(A a) { return a.v; }
  __device__ static Vec zeros() { return Vec{0.0, 0.0}; }
  __device__ static void fmas(Vec& d, const Vec* x, Vec y) {
    d.lo = ::fma(x[1].lo, y.hi, ::fma(x[0].lo, y.lo, d.lo));
    d.hi = ::fma(x[1].hi, y.hi, ::fma(x[0].hi, y.lo, d.hi));
  }
};

template <typename T>
struct Blk {
  T* P;          // slice, column-major, column stride rs, rows >= nr zero
  int rs, rpc;   // rpc: rows of the slice (a multiple of 8)
  T* W;          // [S * bk + bk] reduced sums
  T* Y;          // [bk][SY] minus the solved rows of R, by column
  T* red;        // [kNT]
  Xch x;
};

// W[i * w + a] = sum over this CTA's rows of p_{jx+i} p_{a0+a}, i < n <= S, a < w.  A
// thread forms 4 x 4 entries (i = ii + (S/4) k, a = ai + na k, so that neighbouring lanes read
// neighbouring columns); ks neighbouring lanes share a tile's rows in turns of 16 bytes and are
// combined by exchanges that halve the entries each lane keeps.
template <typename T>
__device__ __forceinline__ void gram(const Blk<T>& c, int jx, int n, int a0, int w) {
  constexpr int S = kS<T>;
  using V = Vec<T>;
  const int na = (w + 3) / 4;
  const int ntiles = (S / 4) * na;
  // FP64: at most four lanes, since a lane without rows takes its share of the FP64 pipe too
  int lks = 0;
  while (lks < (sizeof(T) == 4 ? 5 : 2) && (2 << lks) * ntiles <= kNT) ++lks;
  const int ks = 1 << lks;
  const int kg = threadIdx.x & (ks - 1);
  const T* bx = c.P + (size_t)jx * c.rs;
  const T* by = c.P + (size_t)a0 * c.rs;
  const int stride = kNT >> lks;
  for (int t0 = 0; t0 < ntiles; t0 += stride) {  // the same trip count in every thread
    const int t = t0 + (threadIdx.x >> lks);
    const int ii = t % (S / 4), ai = t / (S / 4);
    typename V::A acc[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[i] = V::zero();
    int x[4], y[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {  // entries past the ranges read their last columns
      x[k] = min(ii + (S / 4) * k, n - 1) * c.rs;
      y[k] = min(ai + na * k, w - 1) * c.rs;
    }
    if (t < ntiles) {
#pragma unroll 2
      for (int r = V::N * kg; r < c.rpc; r += V::N * ks) {
        V xv[4], yv[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          xv[k] = V::ld(bx + x[k] + r);
          yv[k] = V::ld(by + y[k] + r);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int a = 0; a < 4; ++a) V::dot(acc[4 * i + a], xv[i], yv[a]);
      }
    }
    T v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = V::sum(acc[i]);
    int cnt = 16, first = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (lks > q) {
        const int h = 8 >> q;
        const bool up = (kg >> q) & 1;
#pragma unroll
        for (int i = 0; i < h; ++i) {
          const T mine = up ? v[i + h] : v[i], other = up ? v[i] : v[i + h];
          v[i] = mine + __shfl_xor_sync(0xffffffffu, other, 1 << q);
        }
        cnt = h;
        first += up ? h : 0;
      }
    if (lks > 4) v[0] += __shfl_xor_sync(0xffffffffu, v[0], 16);
    if (t < ntiles && kg < 16) {
#pragma unroll
      for (int i = 0; i < 16; ++i)
        if (i < cnt) {
          const int ri = ii + (S / 4) * ((first + i) >> 2), ca = ai + na * ((first + i) & 3);
          if (ri < n && ca < w) c.W[ri * w + ca] = v[i];
        }
    }
  }
}

// This CTA's dot products of column jc with columns a0 .. a1-1 into W[a - a0].
template <typename T>
__device__ __forceinline__ void dots(const Blk<T>& c, int jc, int a0, int a1) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const T* pj = c.P + (size_t)jc * c.rs;
  for (int a = a0 + warp; a < a1; a += kNW) {
    const T* pa = c.P + (size_t)a * c.rs;
    T s = T(0);
    for (int r = lane; r < c.rpc; r += 32) s += pa[r] * pj[r];
    s = warp_sum(s);
    if (lane == 0) c.W[a - a0] = s;
  }
}

// Columns jx .. jx+n-1 <- those columns times the transpose of the lower triangular sLi (element
// (a, k) at a * S + k): four threads per row, each every fourth column.  Every thread calls it.
template <typename T>
__device__ __forceinline__ void times_lit(const Blk<T>& c, int jx, int n, const T* sLi) {
  constexpr int S = kS<T>;
  const int quarter = threadIdx.x / (kNT / 4);
  for (int r0 = 0; r0 < c.rpc; r0 += kNT / 4) {
    const int r = r0 + threadIdx.x % (kNT / 4);
    T* p = c.P + (size_t)jx * c.rs + r;
    T out[S / 4];
    if (r < c.rpc) {
      T v[S];
#pragma unroll
      for (int k = 0; k < S; ++k) v[k] = k < n ? p[k * c.rs] : T(0);
#pragma unroll
      for (int i = 0; i < S / 4; ++i) {
        const T* l = sLi + (4 * i + quarter) * S;
        T s = T(0);
#pragma unroll
        for (int k = 0; k < 4 * i + 4; ++k) s += v[k] * l[k];  // zero past the diagonal
        out[i] = s;
      }
    }
    __syncthreads();
    if (r < c.rpc) {
#pragma unroll
      for (int i = 0; i < S / 4; ++i)
        if (4 * i + quarter < n) p[(4 * i + quarter) * c.rs] = out[i];
    }
  }
}

// What follows runs only for nearly dependent columns; not inlined, so that it costs the usual
// path neither registers nor instruction cache.

// Warp 0: the first factor, which covers gd columns, with floored pivots where those are not all of
// them or a row amplifies more than kMaxHard.  Returns the number of leading columns it covers,
// and from bit 8 up those of them that amplify rounding by more than kMaxAmp.
template <typename T>
__device__ __noinline__ unsigned hard_factor(const T* W, int w, int n, int gd, T* sU, T* sLi, T* sD, T* sRow,
                                             T* sFl, const float* sNrm, const int* sExp) {
  constexpr int S = kS<T>;
  const int lane = threadIdx.x & 31;
  float amp = amplification(sLi, sNrm, sExp, n, gd);
  if (gd < n || __any_sync(0xffffffffu, lane > 0 && lane < gd && !(amp <= kMaxHard<T>))) {
    if (lane < S) sFl[lane] = lane < n ? kFloor<T> * W[lane * w + lane] : T(0);
    __syncwarp();
    gd = cholesky<T, true>(W, w, n, sU, sLi, sD, sRow, sFl);
    amp = amplification(sLi, sNrm, sExp, n, gd);
    const unsigned bad = __ballot_sync(0xffffffffu, lane > 0 && lane < gd && !(amp <= kMaxHard<T>));
    if (bad) gd = min(gd, __ffs(bad) - 1);
  }
  return (unsigned)gd | __ballot_sync(0xffffffffu, lane > 0 && lane < gd && amp > kMaxAmp) << 8;
}

// Columns jx .. jx+n-1 <- T with T U = those columns (U upper triangular, element (a, c) at a * S + c;
// 1 / U_cc at sLi[c * S + c]), by substitution: a thread per row.
template <typename T>
__device__ __noinline__ void solve_u(T* P, int rs, int rpc, int n, const T* sU, const T* sLi) {
  constexpr int S = kS<T>;
  for (int r = threadIdx.x; r < rpc; r += kNT) {
    T v[S];
#pragma unroll
    for (int k = 0; k < S; ++k) {
      T x = k < n ? P[k * rs + r] : T(0);
#pragma unroll
      for (int a = 0; a < k; ++a) x -= v[a] * sU[a * S + k];
      v[k] = x * sLi[k * S + k];
      if (k < n) P[k * rs + r] = v[k];
    }
  }
}

// The second factor ends before the sub-block (what is left of a column lies in the span of those
// before it, to rounding): columns n2 .. n1-1 back to T U, from which the column recurrence goes
// on, and minus their rows of R so far, U2 U, into Y.
template <typename T>
__device__ __noinline__ void give_back(T* P, int rs, int rpc, int n1, int n2, const T* sU, const T* sU2, T* Y) {
  constexpr int S = kS<T>, SY = kSY<T>;
  for (int r = threadIdx.x; r < rpc; r += kNT)
    for (int a = n1 - 1; a >= n2; --a) {
      T x = T(0);
      for (int k = 0; k <= a; ++k) x += P[k * rs + r] * sU[k * S + a];
      P[a * rs + r] = x;
    }
  for (int e = threadIdx.x; e < (n1 - n2) * S; e += kNT) {
    const int a = n2 + e / S, i = e % S;
    T x = T(0);
    if (i < n2)
      for (int k = i; k <= a; ++k) x -= sU2[i * S + k] * sU[k * S + a];
    Y[a * SY + i] = x;
  }
}

template <typename T>
__global__ void __launch_bounds__(kNT, 1) k_panel_blk(T* __restrict__ Q, int64_t ldq,
                                                       T* __restrict__ R, int64_t ldr, int64_t M,
                                                       int bk, int rpc, int rs, double tau2,
                                                       unsigned long long* part,
                                                       unsigned long long* fin, int ecap,
                                                       unsigned* epoch, int* status, int col0,
                                                       long long wait_limit) {
  using V = Vec<T>;
  constexpr int S = kS<T>, SY = kSY<T>;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ __align__(16) T sU[S * S], sLi[S * S], sU2[S * S];
  __shared__ __align__(16) T sRow[16 * S], sD[S];
  __shared__ T sFl[S];
  __shared__ float sNrm[S];
  __shared__ int sExp[S];
  __shared__ int sGood;
  __shared__ unsigned sFail, sHard;
  const int G = gridDim.x, g = blockIdx.x, tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  // the slices stay inside the panel's buffers and the sums inside theirs (the same for every
  // CTA: before any exchange)
  CQR_CHECK(ldq >= M && ldr >= bk && rpc % 8 == 0 && rs >= rpc && (int64_t)G * rpc >= M &&
                bk <= kMaxB && (S * bk + bk) * Wire<T>::kWords <= ecap, 501);
  const int64_t row0 = (int64_t)g * rpc;
  const int nr = (int)max((int64_t)0, min((int64_t)rpc, M - row0));
  Blk<T> c;
  c.P = reinterpret_cast<T*>(smraw);
  c.rs = rs;
  c.rpc = rpc;
  c.Y = c.P + (size_t)bk * rs;  // 16-byte aligned: rs and SY are multiples of 16 bytes
  c.W = c.Y + (size_t)SY * bk;
  c.red = c.W + S * bk + bk;
  T* thr = c.red + kNT;  // [bk]
  c.x = Xch{part, fin, ecap, 0u, status, wait_limit};
  const unsigned tags = 5u * (unsigned)bk + 8u;
  if (tid < 16 * S) sRow[tid] = T(0);
  if (!exchange_begin(c.x, epoch, tags)) return;
  const unsigned first = c.x.tag;

  // the slice into shared memory: 16-byte loads (row0, ldq and Q are multiples of 16 bytes),
  // the rows past M zero
  {
    const int nq = rpc / V::N;
    for (int idx = tid; idx < bk * nq; idx += kNT) {
      const int a = idx / nq, r = (idx - a * nq) * V::N;
      const T* src = Q + row0 + r + a * ldq;
      T* dst = c.P + (size_t)a * rs + r;
      if (r + V::N <= nr)
        *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(src);
      else
#pragma unroll
        for (int u = 0; u < V::N; ++u) dst[u] = r + u < nr ? src[u] : T(0);
    }
  }
  __syncthreads();

  const bool icgs = tau2 > 0.0;
  bool ok = true, broke = false;
  int j = 0, w = bk, n = 0, good = 0;
  unsigned fail = 0u, hard = 0u;  // columns that fail the ICGS test, that amplify rounding
  bool second = false;  // the sub-block's second projection (one copy of the code for both)
  while (j < bk) {
    if (!second) {
      w = bk - j;
      n = min(S, w);
    }
    // the second projection's products: with the computed columns (off of them; none without the
    // ICGS test), the sub-block and, if it amplifies rounding, the columns behind it
    const int off = icgs ? j : 0;
    const int nx = second ? good : n, wx = second ? off + (hard ? w : good) : w;
    gram(c, j, nx, second ? j - off : j, wx);
    int E = nx * wx;
    if (j == 0 && icgs && !second) {
      // the squared norms of every column behind the first products
      for (int a = warp; a < bk; a += kNW) {
        const T* pa = c.P + (size_t)a * rs;
        T s = T(0);
        for (int r = lane; r < rpc; r += 32) s += pa[r] * pa[r];
        s = warp_sum(s);
        if (lane == 0) c.W[E + a] = s;
      }
      E += bk;
    }
    ok = exchange<T, kNT>(c.x, c.W, E, c.red);
    if (!ok) break;
    if (second) {
      // T^T T - Z1^T Z1 into red, T -= Q[:, 0:j] Z1 (four threads per row, each every fourth
      // column)
      for (int idx = warp; idx < good * good; idx += kNW) {
        const int i = idx / good, a = idx - i * good;
        if (a < i) continue;
        T s = T(0);
        for (int k = lane; k < off; k += 32) s += c.W[i * wx + k] * c.W[a * wx + k];
        s = warp_sum(s);
        if (lane == 0) c.red[i * S + a] = c.W[i * wx + off + a] - s;
      }
      for (int r0 = 0; r0 < rpc; r0 += kNT / 4) {
        const int r = r0 + tid % (kNT / 4), quarter = tid / (kNT / 4);
        if (r < rpc && off > 0) {
          const T* q = c.P + r;
          T acc[S / 4];
          int z[S / 4];
#pragma unroll
          for (int i = 0; i < S / 4; ++i) {
            acc[i] = T(0);
            z[i] = min(4 * i + quarter, good - 1) * wx;
          }
#pragma unroll 4
          for (int a = 0; a < off; ++a) {
            const T x = q[(size_t)a * rs];
#pragma unroll
            for (int i = 0; i < S / 4; ++i) acc[i] += x * c.W[z[i] + a];
          }
#pragma unroll
          for (int i = 0; i < S / 4; ++i)
            if (4 * i + quarter < good) c.P[(size_t)(j + 4 * i + quarter) * rs + r] -= acc[i];
        }
      }
      __syncthreads();
    } else if (j == 0 && icgs) {
      // v < tau^2 eta with the product in FP64, as v < (that product rounded up to T)
      for (int a = tid; a < bk; a += kNT) thr[a] = round_up_to<T>(tau2 * (double)c.W[n * bk + a]);
      __syncthreads();
    }
    bool near = second;
    if (second && tid < S * S) {
      const int k = tid / S, a = tid % S;
      near = !(k <= a && a < good) || fabs(c.red[tid] - (k == a ? T(1) : T(0))) < kNearI<T>;
    }
    int gd = good;
    if (second && __syncthreads_and(near)) {
      if (tid < S * S) {
        const int k = tid / S, a = tid % S;
        const T x = a < good && k < a ? c.red[tid] : T(0);
        const T x2 = a < good ? T(0.5) * (c.red[a * S + a] - T(1)) : T(0);
        sU2[tid] = k == a ? T(1) + x2 : x;
        sLi[a * S + k] = k == a ? T(1) - x2 : -x;
      }
    } else if (warp == 0) {
      gd = cholesky<T>(second ? c.red : c.W, second ? S : w, nx, second ? sU2 : sU, sLi, sD, sRow);
      if (!second) {
        if (lane < n) {
          int h;
          sNrm[lane] = norm_of(c.W[lane * w + lane], h);
          sExp[lane] = h;
        }
        __syncwarp();
        const float amp = amplification(sLi, sNrm, sExp, n, gd);
        unsigned big = 0u;
        if (gd < n || __any_sync(0xffffffffu, lane > 0 && lane < gd && !(amp <= kMaxAmp))) {
          const unsigned r = hard_factor(c.W, w, n, gd, sU, sLi, sD, sRow, sFl, sNrm, sExp);
          gd = r & 0xff;
          big = r >> 8;
        }
        // the ICGS test, from the panel's second column on
        const bool test = icgs && lane < gd && j + lane > 0;
        const unsigned f = __ballot_sync(0xffffffffu, test && sD[test ? lane : 0] < thr[test ? j + lane : 0]);
        if (lane == 0) {
          sFail = f;
          sHard = big;
        }
      } else {
        // the pivot of a column of which the second projection takes most has lost its digits
        const bool ok2 = lane >= gd || sD[lane] >= T(0.25) * c.W[lane * wx + off + lane];
        const unsigned lost = ~__ballot_sync(0xffffffffu, ok2);
        if (lost) gd = __ffs(lost) - 1;
      }
    }
    if (tid == 0) sGood = gd;
    __syncthreads();
    if (!second) {
      good = sGood;
      fail = sFail;
      hard = sHard;
    }
    const int behind = good;  // the first column behind the sub-block
    if (second) {
      // R[0:j, S] += Z1 U by the CTAs that own the columns
      for (int a = 0; a < good; ++a)
        if ((j + a) % G == g)
          for (int i = tid; i < off; i += kNT) {
            T s = T(0);
            for (int k = 0; k <= a; ++k) s += c.W[k * wx + i] * sU[k * S + a];
            R[i + (int64_t)(j + a) * ldr] += s;
          }
      if (sGood < good) {
        give_back<T>(c.P + (size_t)j * rs, rs, rpc, good, sGood, sU, sU2, c.Y);
        good = sGood;
        second = good > 0;
        __syncthreads();
      }
    }
    if (good > 0) {
      // minus the rows j .. j+good-1 of R, columns j+good .., by columns in Y: four threads
      // (of four warps) per column, S / 4 rows each
      if (second || !hard) {
        constexpr int H = S / 4;
        const int quarter = tid / (kNT / 4);
        // right-hand sides: the products with P_S or, if the first factor amplifies rounding, with T;
        // else, in the second projection, the rows solved with the first factor (signs: Y's)
        const bool y = second && !hard;
        const T* src = y ? c.Y : c.W + (second ? off : 0);
        const int ss = y ? 1 : wx, sa = y ? SY : 1;
        const T sg = y ? T(1) : T(-1);
        for (int a0 = behind; a0 < w; a0 += kNT / 4) {
          const int a = a0 + tid % (kNT / 4);
          T q[H];
#pragma unroll
          for (int i = 0; i < H; ++i) q[i] = T(0);
          if (a < w)
#pragma unroll 1
            for (int m = 0; m <= quarter; ++m) {
              T x[H];
#pragma unroll
              for (int i = 0; i < H; ++i) {
                const int k = m * H + i;
                x[i] = k < good ? src[k * ss + a * sa] : T(0);
              }
#pragma unroll
              for (int i = 0; i < H; ++i) {
                const T* l = sLi + (quarter * H + i) * S + m * H;  // zero past the diagonal
#pragma unroll
                for (int u = 0; u < H; ++u) q[i] += x[u] * l[u];
              }
            }
          __syncthreads();
          if (a < w)
#pragma unroll
            for (int i = 0; i < H; ++i)
              c.Y[a * SY + quarter * H + i] = quarter * H + i < good ? sg * q[i] : T(0);
        }
      }
      // T = P_S U^{-1}; then Q_S = T U2^{-1}
      if (hard && !second)
        solve_u<T>(c.P + (size_t)j * rs, rs, rpc, good, sU, sLi);
      else
        times_lit(c, j, good, sLi);
      __syncthreads();
      if ((fail | hard) && !second) {
        second = true;
        continue;
      }
      if (second) {
        // U <- U2 U
        if (tid < S * S) {
          const int i = tid / S, a = tid % S;
          T s = T(0);
          if (i <= a && a < good)
            for (int k = i; k <= a; ++k) s += sU2[i * S + k] * sU[k * S + a];
          c.red[tid] = s;
        }
        __syncthreads();
        if (tid < S * S) sU[tid] = c.red[tid];
        if (g == 0 && tid == 0 && icgs) {
          int count = __popc(fail & ((1u << good) - 1u));
          if (hard) {  // by R's diagonal, since the first pivots miss what a raised one takes
            count = 0;
            for (int a = 0; a < good; ++a) count += j + a > 0 && c.red[a * S + a] * c.red[a * S + a] < thr[j + a];
          }
          if (count) atomicAdd(status + ST_REORTH, count);
        }
        __syncthreads();
        second = false;
      }
      // R: column j+a is written by CTA (j+a) mod G
      for (int a = (g + G - j % G) % G; a < w; a += G)
        if (tid < good && tid <= a)
          R[j + tid + (int64_t)(j + a) * ldr] = a < good ? sU[tid * S + a] : -c.Y[a * SY + tid];
      // P -= Q_S R_rest: a thread takes 16 bytes of rows of eight columns
      const int nq = rpc / V::N, nc8 = (w - good + 7) / 8;
      for (int t = tid; t < nq * nc8; t += kNT) {
        const int cg = t / nq, r = (t - cg * nq) * V::N;
        const int a0 = good + 8 * cg;
        const T* q = c.P + (size_t)j * rs + r;
        T* p = c.P + (size_t)(j + a0) * rs + r;
        V acc[8];
        const int nv = min(8, w - a0);
#pragma unroll
        for (int u = 0; u < 8; ++u) acc[u] = V::ld(p + (size_t)min(u, nv - 1) * rs);
        const T* y = c.Y + (size_t)a0 * SY;
#pragma unroll 2
        for (int k = 0; k < S; k += V::N) {
          V qv[V::N];
#pragma unroll
          for (int i = 0; i < V::N; ++i) qv[i] = k + i < good ? V::ld(q + (size_t)(k + i) * rs) : V::zeros();
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const V yu = V::ld(y + (size_t)min(u, nv - 1) * SY + k);
            V::fmas(acc[u], qv, yu);
          }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (u < nv) V::st(p + (size_t)u * rs, acc[u]);
      }
      j += good;
      __syncthreads();
    }
    if (good == n) continue;
    // column j by the column recurrence: its products; when the ICGS test asks for it, its
    // products with the computed columns, the projection on them, and its products again
    for (int pass = 0;; ++pass) {
      dots(c, j, pass == 1 ? 0 : j, pass == 1 ? j : bk);
      ok = exchange<T, kNT>(c.x, c.W, pass == 1 ? j : bk - j, c.red);
      if (!ok || pass == 2) break;
      if (pass == 0 && !(j > 0 && icgs && c.W[0] < thr[j])) break;
      if (pass == 1) {
        for (int r = tid; r < rpc; r += kNT) {
          T acc = c.P[(size_t)j * rs + r];
          for (int a = 0; a < j; ++a) acc -= c.P[(size_t)a * rs + r] * c.W[a];
          c.P[(size_t)j * rs + r] = acc;
        }
        if (j % G == g)
          for (int a = tid; a < j; a += kNT) R[a + (int64_t)j * ldr] += c.W[a];
        if (g == 0 && tid == 0) atomicAdd(status + ST_REORTH, 1);
      }
      __syncthreads();  // W is read, column j written
    }
    if (!ok) break;
    const T v0 = c.W[0];
    if (!(v0 > T(0)) || !isfinite(v0)) {
      if (g == 0 && tid == 0) set_status(status, CQR_EBREAKDOWN, col0 + j);
      broke = true;
      break;
    }
    const T rjj = sqrt(v0);
    const T inv = T(1) / rjj;
    for (int a = tid; a < bk - j; a += kNT)
      if ((j + a) % G == g) R[j + (int64_t)(j + a) * ldr] = a == 0 ? rjj : c.W[a] * inv;
    for (int r = tid; r < rpc; r += kNT) {
      T* p = c.P + (size_t)j * rs + r;
      const T q = *p * inv;
      *p = q;
      for (int a = 1; a < bk - j; ++a) p[(size_t)a * rs] -= q * (c.W[a] * inv);
    }
    ++j;
    __syncthreads();
  }
  exchange_end(epoch, first, tags);
  if (!ok || broke) return;
  {
    const int nq = rpc / V::N;
    for (int idx = tid; idx < bk * nq; idx += kNT) {
      const int a = idx / nq, r = (idx - a * nq) * V::N;
      T* dst = Q + row0 + r + a * ldq;
      const T* src = c.P + (size_t)a * rs + r;
      if (r + V::N <= nr)
        *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(src);
      else
#pragma unroll
        for (int u = 0; u < V::N; ++u)
          if (r + u < nr) dst[u] = src[u];
    }
  }
}

template <typename T>
size_t blk_smem(int bk, int rs) {
  return ((size_t)bk * rs + (size_t)kS<T> * bk + bk + (size_t)kSY<T> * bk + kNT + bk) * sizeof(T) + 64;
}

size_t blk_words(int bk, size_t elem) {
  return (size_t)((elem == 4 ? kS<float> : kS<double>) * bk + bk) * (elem / 4);
}

}  // namespace

// Rows per CTA.  FP32: 128 where that fits shared memory and the SMs.  More CTAs than that gain
// nothing (a column costs its exchanges: 5120 x 128 takes 96 us per panel at 128 rows, 101 at
// 40, 116 at 192), and they keep panels of other streams out (16 problems of 9216 x 128 panels on
// 16 streams, forward and adjoint: 54 ms at 128 rows, 78 at 64).  FP64: 24, since the
// FP64 pipes are slow and every SM's are wanted.  Otherwise as few rows as the SMs allow.
// Column stride congruent to 32 bytes mod 64 (gram's bank pattern).
bool plan_panel_blk(int64_t M, int bk, size_t elem, int num_sms, PanelBlkPlan* p) {
  const char* env = getenv("CQR_PANEL_BLK");
  if (env && env[0] == '0') return false;
  if (bk > kMaxB) return false;
  const int64_t least = (M + num_sms - 1) / num_sms;
  const int64_t want[2] = {std::max<int64_t>(least, elem == 4 ? 128 : 24), least};
  for (int64_t rpc : want) {
    rpc = (rpc + 7) / 8 * 8;
    if (rpc > 4096) continue;
    const int unit = (int)(64 / elem), half = unit / 2;  // elements of 64 and 32 bytes
    int rs = (int)rpc;
    while (rs % unit != half) rs += half;
    const size_t sm = elem == 4 ? blk_smem<float>(bk, rs) : blk_smem<double>(bk, rs);
    if (sm + 8 * 1024 > kSmemCap) continue;
    p->rpc = (int)rpc;
    p->rs = rs;
    p->G = (int)((M + rpc - 1) / rpc);
    p->smem_bytes = sm;
    return true;
  }
  return false;
}

size_t panel_blk_bytes(int bk, size_t elem, int num_sms) {
  if (bk > kMaxB) return 256;
  return 256 + (size_t)(num_sms + 1) * blk_words(bk, elem) * sizeof(u64);
}

// ws: panel_blk_bytes bytes (zero before the first launch): the tag count, the sums, the partials.
template <typename T>
cudaError_t launch_panel_blk(const PanelBlkPlan& p, T* Q, int64_t ldq, T* R, int64_t ldr, int64_t M,
                             int bk, double tau, void* ws, int* status, int col0, cudaStream_t st,
                             long long wait_limit) {
  const void* fn = (const void*)k_panel_blk<T>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)p.smem_bytes);
  if (e != cudaSuccess) return e;
  double tau2 = tau > 0.0 ? tau * tau : -1.0;
  long long wl = wait_limit > 0 ? wait_limit : kWaitLimitCycles;
  int rpc = p.rpc, rs = p.rs;
  int ecap = (int)blk_words(bk, sizeof(T));
  unsigned* epoch = static_cast<unsigned*>(ws);
  u64* fin = reinterpret_cast<u64*>(static_cast<char*>(ws) + 256);
  u64* part = fin + ecap;
  void* args[] = {&Q, &ldq, &R, &ldr, &M, &bk, &rpc, &rs, &tau2, &part, &fin, &ecap, &epoch,
                  &status, &col0, &wl};
  return cudaLaunchCooperativeKernel(fn, dim3(p.G), dim3(kNT), args, p.smem_bytes, st);
}

template cudaError_t launch_panel_blk<float>(const PanelBlkPlan&, float*, int64_t, float*, int64_t,
                                             int64_t, int, double, void*, int*, int, cudaStream_t,
                                             long long);
template cudaError_t launch_panel_blk<double>(const PanelBlkPlan&, double*, int64_t, double*,
                                              int64_t, int64_t, int, double, void*, int*, int,
                                              cudaStream_t, long long);

cudaError_t bounds_take_panel_blk(int* code, int* site) { return bounds_take_here(code, site); }

}  // namespace cqr
