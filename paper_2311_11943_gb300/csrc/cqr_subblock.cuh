// cqr_subblock.cuh -- the small factorisation of a sub-block of panel columns, shared by the panel of
// a single problem (cqr_panel_blk.cu) and of a batch (cqr_batched.cu).
#pragma once
#include "cqr_device.cuh"

namespace cqr {

// Columns per sub-block: 16 in FP32; 8 in FP64, whose S x S factor would not stay in registers.
template <typename T>
constexpr int kS = sizeof(T) == 4 ? 16 : 8;
// Rows of U^{-T} that amplify rounding by more than this (the sum over k of |U^{-T}_ak| |p_k|, 1 for
// orthogonal columns) are not used as they are: a batch cuts the sub-block there, a single
// problem's panel projects it a second time.
constexpr float kMaxAmp = 4.0f;

// 1 / sqrt(d) for positive finite d from an FP32 estimate y of relative error e / 2, where
// e = 1 - d y^2: y (1 + e / 2) in FP32, y (1 + e / 2 + 3 e^2 / 8) in FP64 (the next term of the
// binomial series is below 2^-66).  In FP64 the estimate is of the significand with an even
// exponent, so that it neither overflows nor underflows; the FP64 pipe is slow, so no more
// operations than these.
__device__ __forceinline__ float inv_root(float d) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(d));
  return fmaf(0.5f * y, fmaf(-(d * y), y, 1.f), y);
}
__device__ __forceinline__ double inv_root(double d) {
  const long long b = __double_as_longlong(d);
  const int h = ((int)(b >> 52) - 1023) >> 1;  // d = m 4^h, 1 <= m < 4
  const double m = __longlong_as_double(b - ((long long)(2 * h) << 52));
  const double y = (double)rsqrtf((float)m);
  const double e = fma(-(m * y), y, 1.0);
  const double r = fma(y, e * fma(0.375, e, 0.5), y);
  return __longlong_as_double(__double_as_longlong(r) - ((long long)h << 52));
}
// Whether d is a pivot that inv_root takes: positive, normal, finite (by its bits, so that the
// FP64 pipe is left alone), and small enough that no square of a scaled entry overflows.
__device__ __forceinline__ bool fine_pivot(float d) {
  const int b = __float_as_int(d);
  return b >= 0x00800000 && b < 0x7f000000;
}
__device__ __forceinline__ bool fine_pivot(double d) {
  const int hi = __double2hiint(d);
  return hi >= 0x00200000 && hi < 0x7fc00000;
}

// Cholesky of an n x n block (n <= S; element (i, a), i <= a, at B[i * ld + a]) by warp 0 with
// the identity beside it: lane a < S holds column a, lane S + c column c of the identity.  Bound
// by latency, so four rows per turn: they go round through shared memory, every lane factors
// their 4 x 4 diagonal block for itself and solves its own column, the solved rows go round, are
// taken off the rows behind, and those move up by four registers (one rolled loop: straight-line
// code that runs once per sub-block waits for its instructions).  U into sU[k * S + a] (k <= a),
// U^{-T} into sLi[k * S + c] (zero for c > k), the pivots into sD; sRow: [2][2 S][4].  FLOOR: the
// pivot of column k is fl[k] where it is less (fl[S], zero from n).  Returns the number of leading
// columns with a fine pivot.
template <typename T, bool FLOOR = false>
__device__ __forceinline__ int cholesky(const T* B, int ld, int n, T* sU, T* sLi, T* sD, T* sRow,
                                        const T* fl = nullptr) {
  constexpr int S = kS<T>;
  const int lane = threadIdx.x & 31;
  T* raw = sRow;              // rows as they stand, [column][4]
  T* done = sRow + 2 * S * 4;  // solved rows; entries past column S are read into unused rows
  T col[S];
#pragma unroll
  for (int k = 0; k < S; ++k)
    col[k] = lane < n ? (k <= lane ? B[k * ld + lane] : T(0)) : (lane - S == k ? T(1) : T(0));
  int good = n;
#pragma unroll 1
  for (int k = 0; k < S; k += 4) {
    if (lane < S)
#pragma unroll
      for (int q = 0; q < 4; ++q) raw[lane * 4 + q] = col[q];
    __syncwarp();
    T m[4][4], iv[4], d[4], u[4];
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int q = 0; q < 4; ++q) m[q][p] = raw[(k + p) * 4 + q];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      d[q] = m[q][q];
      if constexpr (FLOOR) d[q] = d[q] < fl[k + q] ? fl[k + q] : d[q];
      // rows behind a bad pivot hold rubbish and are not used
      good = k + q < good && !fine_pivot(d[q]) ? k + q : good;
      iv[q] = inv_root(d[q]);
#pragma unroll
      for (int p = q + 1; p < 4; ++p) m[q][p] *= iv[q];
#pragma unroll
      for (int i = q + 1; i < 4; ++i)
#pragma unroll
        for (int p = i; p < 4; ++p) m[i][p] -= m[q][i] * m[q][p];
      T x = col[q];
#pragma unroll
      for (int i = 0; i < q; ++i) x -= m[i][q] * u[i];
      u[q] = x * iv[q];
      if constexpr (FLOOR)
        if (lane == k + q) u[q] = d[q] * iv[q];
    }
    if (lane < S)
#pragma unroll
      for (int q = 0; q < 4; ++q) done[lane * 4 + q] = u[q];
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (lane < S) {
        if (lane >= k + q) sU[(k + q) * S + lane] = u[q];
      } else if (lane < 2 * S) {
        sLi[(k + q) * S + lane - S] = lane - S <= k + q ? u[q] : T(0);
      }
      if (lane == 0) sD[k + q] = d[q];
    }
#pragma unroll
    for (int i = 4; i < S; ++i) {
      T x = col[i];
#pragma unroll
      for (int q = 0; q < 4; ++q) x -= done[(k + i) * 4 + q] * u[q];
      col[i - 4] = x;
    }
  }
  __syncwarp();
  return good;
}

}  // namespace cqr
