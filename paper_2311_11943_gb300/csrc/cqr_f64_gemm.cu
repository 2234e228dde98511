// cqr_f64_gemm.cu -- the FP64 trailing update (a4, a5) on the BF16 tensor cores, by exact integer
// slices (Ozaki, Ogita, Oishi and Rump 2012; on tensor cores Mukunoki et al. 2020):
//   GEMM1  Rbar = Qbar^T B            (K = all M rows)
//   GEMM2  C -= Qbar Rbar             (K = the panel width)
//
// Each operand vector along K (a column of Qbar and of B, a row of Qbar, a column of Rbar) is
// scaled by the power of two above its largest magnitude and rounded to a 56-bit integer, which
// is cut into seven signed 8-bit digits, most significant first: exact BF16 values.  A product of
// two numbers is sum over (i, j) of digit products of weight 256^-(i+j); the pairs of equal
// i + j = g < 7 are summed in one FP32 accumulator, exactly, since 256 products of two 7-bit
// magnitudes times the at most four pairs that have to be exact stay below 2^24 (the sums of g > 3
// may round, when all of their digits are near the largest: by a unit of their group, for g = 4
// 2^-46 of one product of the largest magnitudes and 2^-54 of the sum of 256 of them).  Every 256 of K the seven accumulators are read, converted
// and added up, exactly, in one 76-bit integer per output (64 bits in units of 2^12 and a 16-bit
// remainder), which becomes a double once, at the end.  What is lost are the dropped pairs
// (g >= 7) and the rounding of the operands, each below 2^-53 of a product of the largest
// magnitudes, and the final rounding.  An infinite or NaN entry makes its row or column of the
// product NaN.  Against products in quadruple precision (rms over entries, relative to the norms
// of the factors for GEMM1, to |C| + |Qbar| |Rbar| for GEMM2; CUDA cores, then this):
//   N(0,1) 3000 x 480 by 32         1.2e-17, 3.9e-17   5.6e-18, 3.6e-17
//   N(0,1) 4100 x 272 by 128        1.2e-17, 4.0e-17   5.3e-18, 2.6e-17
//   columns over 16 decades         1.2e-17, 3.9e-17   7.1e-18, 3.6e-17
//   rows over 8 decades             4.6e-17, 4.1e-17   6.3e-17, 3.4e-17
//
// Why: GB300's FP64 pipes give 1.2 TFLOP/s (both GEMMs ran at 1.0 to 1.2), its BF16 tensor
// cores about 1900 in 28 products: 4096 x 4096, b = 128, both GEMMs 231 ms per run on the CUDA
// cores, 20 this way (digits included).  One CTA per 128 x 64 output tile: seven accumulators of 64 columns take 448 of the
// 512 TMEM columns.  Stages of 64 of K: the seven A tiles (16 KB each) have a barrier of their
// own each, so that tile i of the next stage loads as soon as the products of digit i are done;
// the seven B tiles (8 KB each) are double-buffered.  Warps as in cqr_tc_gemm.cu: producer, MMA
// issuer, two idle, eight epilogue warps.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <new>

#include "coded_qr.h"
#include "cqr_device.cuh"
#include "cqr_kernels.cuh"
#include "cqr_umma.cuh"

namespace cqr {

namespace {

using namespace umma;

constexpr int kD = 7;            // digits
constexpr int BM = 128, BN = 64;
constexpr int BK = 64;           // K of a stage: one 128-byte swizzle row of BF16
constexpr int kChunk = 4;        // stages between two readings of the accumulators (K = 256)
constexpr int kEpiWarps = 8;
constexpr int kThreads = 32 * (4 + kEpiWarps);
constexpr uint32_t kBytesA = BM * 128, kBytesB = BN * 128;
constexpr uint32_t kSmemB = kD * kBytesA;
constexpr uint32_t kSmemTiles = kSmemB + 2 * kD * kBytesB;
constexpr uint32_t kSmemTotal = kSmemTiles + 1024 + 256;
constexpr int kUnit = 12;        // the 64-bit sums count 2^kUnit products of the last group
// K of a work unit: 2^14 kMaxK products of weight 2^(48 - kUnit) below 2^63, and kMaxK / 256
// remainders below 2^kUnit within 16 bits
constexpr int kMaxK = 4096;
constexpr int kNone = 1 << 30;   // exponent of a vector with an infinite or NaN entry

struct OzJob {
  int epi;                 // 0: store partial sums; 1: C -= D
  int m_tiles, n_tiles, splits;
  int kp_a, kp_b;          // K stride between the digit planes of A and B (elements)
  int64_t K, kchunk;       // K, K per split (multiples of BK)
  int64_t mrows, ncols;
  const int* ea;           // exponents of A's rows and B's columns
  const int* eb;
  double* out;
  int64_t ldo, split_stride;
  int* status;
};

constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                            ((uint32_t)(BM >> 4) << 24);

__device__ __forceinline__ void mma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d), "l"(a), "l"(b), "r"(kIdesc), "r"(accum)
      : "memory");
}

// Eight TMEM columns of this warp's 32 lanes; the caller waits (tmem_wait) before it uses them.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                 "=r"(r[7])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// a 2^s as a double, rounded to nearest (halves away from zero), by integer operations; zero
// below the normal range, infinite above it.
__device__ __forceinline__ double scaled(long long a, int s) {
  if (a == 0) return 0.0;
  const unsigned long long sign = (unsigned long long)a & 0x8000000000000000ull;
  unsigned long long m = a < 0 ? 0ull - (unsigned long long)a : (unsigned long long)a;
  const int lz = __clzll((long long)m);
  m <<= lz;  // 1 <= m 2^-63 < 2
  int e = 63 - lz + s + 1023;
  const unsigned long long up = m + 0x400ull;
  if (up < m) {
    ++e;
    m = 0x8000000000000000ull;
  } else {
    m = up;
  }
  if (e < 1) return __longlong_as_double((long long)sign);
  if (e > 2046) return __longlong_as_double((long long)(sign | 0x7ff0000000000000ull));
  return __longlong_as_double((long long)(sign | (((unsigned long long)(e - 1) << 52) + (m >> 11))));
}

// (a + r 2^-kUnit) 2^s, 0 <= r < 2^16.
__device__ __forceinline__ double scaled2(long long a, unsigned r, int s) {
  a += r >> kUnit;
  r &= (1u << kUnit) - 1u;
  const int room = __clzll(a < 0 ? ~a : a) - 1;
  const int sh = room < kUnit ? room : kUnit;
  return scaled((long long)((unsigned long long)a << sh) + (r >> (kUnit - sh)), s - sh);
}

__global__ void __launch_bounds__(kThreads, 1) k_f64_gemm(const __grid_constant__ CUtensorMap ma,
                                                           const __grid_constant__ CUtensorMap mb,
                                                           const OzJob job) {
  extern __shared__ __align__(1024) unsigned char smraw[];
  const uint32_t base_u = su32(smraw);
  const uint32_t tiles_u = (base_u + 1023u) & ~1023u;
  unsigned char* tiles = smraw + (tiles_u - base_u);
  uint64_t* full_a = reinterpret_cast<uint64_t*>(tiles + kSmemTiles);  // [kD]
  uint64_t* empty_a = full_a + kD;                                     // [kD]
  uint64_t* full_b = empty_a + kD;                                     // [2]
  uint64_t* empty_b = full_b + 2;                                      // [2]
  uint64_t* acc_full = empty_b + 2;
  uint64_t* acc_empty = acc_full + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // the output tiles stay inside `out` (uniform over the launch: before any barrier)
  CQR_CHECK(job.ldo >= job.mrows && (int64_t)job.m_tiles * BM >= job.mrows &&
                (int64_t)job.n_tiles * BN >= job.ncols && job.kchunk <= kMaxK &&
                job.kchunk * job.splits >= job.K && job.K <= job.kp_a && job.K <= job.kp_b, 701);
  const int total = job.m_tiles * job.n_tiles * job.splits;

  if (threadIdx.x == 0) {
    for (int i = 0; i < kD; ++i) {
      mbar_init(&full_a[i], 1);
      mbar_init(&empty_a[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&full_b[i], 1);
      mbar_init(&empty_b[i], 1);
    }
    mbar_init(acc_full, 1);
    mbar_init(acc_empty, kEpiWarps);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    prefetch_tmap(&ma);
    prefetch_tmap(&mb);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     su32(tmem_slot)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  auto stages = [&](int split) -> int {
    const int64_t k0 = (int64_t)split * job.kchunk;
    const int64_t k1 = k0 + job.kchunk < job.K ? k0 + job.kchunk : job.K;
    return k1 > k0 ? (int)((k1 - k0 + BK - 1) / BK) : 0;
  };

  if (warp == 0) {
    if (lane == 0) {
      int it = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < total && ok; t += gridDim.x) {
        const int split = t % job.splits, mn = t / job.splits;
        const int mt = mn % job.m_tiles, nt = mn / job.m_tiles;
        const int nk = stages(split);
        for (int kb = 0; kb < nk && ok; ++kb, ++it) {
          const int x = (int)((int64_t)split * job.kchunk) + kb * BK;
          const int s = it & 1;
          if (!(ok = mbar_wait(&empty_b[s], ((it >> 1) & 1) ^ 1, abort_flag))) break;
          mbar_expect_tx(&full_b[s], kD * kBytesB);
          for (int p = 0; p < kD; ++p)
            tma_load_2d(tiles_u + kSmemB + (s * kD + p) * kBytesB, &mb, p * job.kp_b + x, nt * BN,
                        &full_b[s]);
          for (int p = 0; p < kD; ++p) {
            if (!(ok = mbar_wait(&empty_a[p], (it & 1) ^ 1, abort_flag))) break;
            mbar_expect_tx(&full_a[p], kBytesA);
            tma_load_2d(tiles_u + p * kBytesA, &ma, p * job.kp_a + x, mt * BM, &full_a[p]);
          }
        }
      }
      // the last loads have landed before the CTA may exit (bounded; after an abandoned wait,
      // those that were issued)
      if (ok) {
        for (int i = it > 1 ? it - 2 : 0; i < it; ++i) {
          const long long t0 = clock64();
          while (!mbar_test(&full_b[i & 1], (i >> 1) & 1) && clock64() - t0 < kWaitLimitCycles) {
          }
        }
        for (int p = 0; p < kD && it > 0; ++p) {
          const long long t0 = clock64();
          while (!mbar_test(&full_a[p], (it - 1) & 1) && clock64() - t0 < kWaitLimitCycles) {
          }
        }
      } else {
        const long long t0 = clock64();
        while (clock64() - t0 < 10 * kDrainCycles) {
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      int it = 0, ch = 0;  // stages, accumulator fills
      bool ok = true;
      for (int t = blockIdx.x; t < total && ok; t += gridDim.x) {
        const int nk = stages(t % job.splits);
        for (int kb = 0; kb < nk && ok; ++kb, ++it) {
          const bool first = kb % kChunk == 0;
          if (first && !(ok = mbar_wait(acc_empty, (ch & 1) ^ 1, abort_flag))) break;
          const int s = it & 1;
          if (!(ok = mbar_wait(&full_b[s], (it >> 1) & 1, abort_flag))) break;
          tc_fence_after();
#pragma unroll 1
          for (int i = 0; i < kD; ++i) {
            if (!(ok = mbar_wait(&full_a[i], it & 1, abort_flag))) break;
            tc_fence_after();
            const uint32_t a = tiles_u + i * kBytesA;
#pragma unroll 1
            for (int j = 0; j < kD - i; ++j) {
              const uint32_t b = tiles_u + kSmemB + (s * kD + j) * kBytesB;
              const uint32_t d = tmem + (uint32_t)((i + j) * BN);
#pragma unroll
              for (int ks = 0; ks < BK / 16; ++ks)
                // a group's first product of a fill is that of digits (0, g)
                mma_bf16(d, sdesc(a + ks * 32), sdesc(b + ks * 32), first && i == 0 && ks == 0 ? 0u : 1u);
            }
            mma_commit(&empty_a[i]);
          }
          if (!ok) break;
          mma_commit(&empty_b[s]);
          if (kb % kChunk == kChunk - 1 || kb == nk - 1) {
            mma_commit(acc_full);
            ++ch;
          }
        }
      }
    }
  } else if (warp >= 4) {
    // epilogue: TMEM lanes 32 (warp % 4) .. +32, columns 32 half .. +32 of every accumulator
    const int ew = warp & 3, half = (warp - 4) >> 2;
    int ch = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < total && ok; t += gridDim.x) {
      const int split = t % job.splits, mn = t / job.splits;
      const int mt = mn % job.m_tiles, nt = mn / job.m_tiles;
      const int nk = stages(split);
      long long acc[32];
      unsigned rem[16];  // remainders of columns 2 i (low half) and 2 i + 1
#pragma unroll
      for (int i = 0; i < 32; ++i) acc[i] = 0;
#pragma unroll
      for (int i = 0; i < 16; ++i) rem[i] = 0u;
      for (int kb = 0; kb < nk; kb += kChunk, ++ch) {
        if (!(ok = mbar_wait(acc_full, ch & 1, abort_flag))) break;
        tc_fence_after();
        const uint32_t lanes = tmem + ((uint32_t)(ew * 32) << 16) + (uint32_t)(half * 32);
#pragma unroll
        for (int c8 = 0; c8 < 4; ++c8) {
          uint32_t r[kD][8];
#pragma unroll
          for (int g = 0; g < kD; ++g) tmem_ld8(lanes + g * BN + c8 * 8, r[g]);
          tmem_wait();
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            int v[kD];
#pragma unroll
            for (int g = 0; g < kD; ++g) v[g] = __float2int_rn(__uint_as_float(r[g][q]));
            // weights 2^(8 (6 - g)), of acc 2^12; |v0| <= 2^22, so v0 256 + v1 fits 32 bits
            const long long lo = (long long)v[4] * (1 << 16) + (long long)v[5] * (1 << 8) + v[6];
            long long a = acc[c8 * 8 + q] + (lo >> kUnit);
            a += (long long)(v[0] * 256 + v[1]) * (1 << 28);
            a += (long long)v[2] * (1 << 20);
            a += (long long)v[3] * (1 << 12);
            acc[c8 * 8 + q] = a;
            rem[c8 * 4 + q / 2] += ((unsigned)lo & 0xfffu) << (q & 1 ? 16 : 0);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty);
      }
      if (!ok) break;
      // value = acc 2^kUnit 2^(ea - 55) 2^(eb - 55) 2^48
      const int64_t row = (int64_t)mt * BM + ew * 32 + lane;
      const bool row_ok = row < job.mrows;
      const int ea = row_ok ? job.ea[row] : 0;
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const int64_t col = (int64_t)nt * BN + half * 32 + i;
        if (!row_ok || col >= job.ncols) continue;
        const int eb = job.eb[col];
        const double v = ea == kNone || eb == kNone ? nan_value<double>()
                                                    : scaled2(acc[i], (rem[i / 2] >> (i & 1 ? 16 : 0)) & 0xffffu,
                                                              ea + eb + kUnit + 48 - 110);
        double* o = job.out + (int64_t)split * job.split_stride + row + col * job.ldo;
        if (job.epi == 0)
          *o = v;
        else
          *o -= v;
      }
    }
  }

  __syncthreads();
  if (*abort_flag && threadIdx.x == 0) set_status(job.status, CQR_ETIMEOUT, 21);
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u)
                 : "memory");
  }
}

// ------------------------------------------------------------------ operand digits
// Exponent e of a largest magnitude: |x| < 2^e (0 for zero), from its high word without the sign.
__device__ __forceinline__ int exp_above(int hi) {
  const int ex = hi >> 20;
  return ex == 0x7ff ? kNone : hi == 0 ? 0 : (ex > 1 ? ex : 1) - 1022;
}

// x 2^(55 - e) rounded to an integer (|x| < 2^e).
__device__ __forceinline__ long long fixed55(double x, int e) {
  const long long b = __double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  unsigned long long m = (unsigned long long)b & 0xfffffffffffffull;
  if (ex) m |= 0x10000000000000ull;
  const int sh = (ex ? ex : 1) - 1075 + 55 - e;  // at most 2
  unsigned long long v;
  if (sh >= 0)
    v = m << sh;
  else if (sh > -56)
    v = (m + (1ull << (-sh - 1))) >> (-sh);
  else
    v = 0ull;
  return b < 0 ? -(long long)v : (long long)v;
}

// The seven digits of v, most significant first, as BF16 bits.
__device__ __forceinline__ void digits(long long v, unsigned short* d) {
#pragma unroll
  for (int p = kD - 1; p > 0; --p) {
    const int c = (int)(signed char)(v & 0xff);
    d[p] = __bfloat16_as_ushort(__int2bfloat16_rn(c));
    v = (v - c) >> 8;
  }
  d[0] = __bfloat16_as_ushort(__int2bfloat16_rn((int)v));
}

// Columns of X (K x n, column-major): one CTA per column, digit planes at out[col][p][kp], zero
// from K to kend (a multiple of 64), exponents e[col].
__global__ void __launch_bounds__(256) k_f64_digits_cols(const double* __restrict__ X, int64_t ldx,
                                                         int64_t K, int64_t kend, int64_t kp,
                                                         unsigned short* __restrict__ out,
                                                         int* __restrict__ e) {
  CQR_CHECK(ldx >= K && kend <= kp, 702);
  __shared__ int s[8];
  const int tid = threadIdx.x;
  const double* x = X + (int64_t)blockIdx.x * ldx;
  int hi = 0;
  for (int64_t k = tid; k < K; k += 256) hi = max(hi, __double2hiint(x[k]) & 0x7fffffff);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  if ((tid & 31) == 0) s[tid >> 5] = hi;
  __syncthreads();
  for (int k = 0; k < 8; ++k) hi = max(hi, s[k]);
  // a largest magnitude whose high word is zero: below 2^-1042, an exponent of -1021 covers it
  const int ex = hi == 0 ? -1021 : exp_above(hi);
  if (tid == 0) e[blockIdx.x] = ex;
  const int es = ex == kNone ? 1025 : ex;
  unsigned short* o = out + (int64_t)blockIdx.x * kD * kp;
  for (int64_t k = 2 * tid; k < kend; k += 512) {
    unsigned short d0[kD], d1[kD];
    digits(k < K && ex != kNone ? fixed55(x[k], es) : 0ll, d0);
    digits(k + 1 < K && ex != kNone ? fixed55(x[k + 1], es) : 0ll, d1);
#pragma unroll
    for (int p = 0; p < kD; ++p)
      *reinterpret_cast<uint32_t*>(o + p * kp + k) = (uint32_t)d0[p] | ((uint32_t)d1[p] << 16);
  }
}

// Rows of X (M x n, column-major): a CTA takes 32 rows, through shared memory; planes at
// out[row][p][kp], zero from n to kend, exponents e[row].
__global__ void __launch_bounds__(256) k_f64_digits_rows(const double* __restrict__ X, int64_t ldx,
                                                         int64_t M, int n, int kend, int64_t kp,
                                                         unsigned short* __restrict__ out,
                                                         int* __restrict__ e) {
  CQR_CHECK(ldx >= M && kend <= kp, 703);
  __shared__ double t[32][65];
  __shared__ int sh[32][8], se[32];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int64_t r0 = (int64_t)blockIdx.x * 32;
  int hi = 0;
  if (r0 + tx < M)
    for (int k = ty; k < n; k += 8) hi = max(hi, __double2hiint(X[r0 + tx + (int64_t)k * ldx]) & 0x7fffffff);
  sh[tx][ty] = hi;
  __syncthreads();
  if (ty == 0) {
    for (int k = 1; k < 8; ++k) hi = max(hi, sh[tx][k]);
    const int ex = hi == 0 ? -1021 : exp_above(hi);
    se[tx] = ex;
    if (r0 + tx < M) e[r0 + tx] = ex;
  }
  for (int k0 = 0; k0 < kend; k0 += 64) {
    __syncthreads();
    for (int k = ty; k < 64; k += 8)
      t[tx][k] = (r0 + tx < M && k0 + k < n) ? X[r0 + tx + (int64_t)(k0 + k) * ldx] : 0.0;
    __syncthreads();
    for (int r = ty; r < 32; r += 8) {
      if (r0 + r >= M) continue;
      const int ex = se[r];
      const int es = ex == kNone ? 1025 : ex;
      unsigned short d0[kD], d1[kD];
      digits(ex == kNone ? 0ll : fixed55(t[r][2 * tx], es), d0);
      digits(ex == kNone ? 0ll : fixed55(t[r][2 * tx + 1], es), d1);
      unsigned short* o = out + (r0 + r) * kD * kp + k0 + 2 * tx;
#pragma unroll
      for (int p = 0; p < kD; ++p)
        *reinterpret_cast<uint32_t*>(o + p * kp) = (uint32_t)d0[p] | ((uint32_t)d1[p] << 16);
    }
  }
}

int64_t up64(int64_t x) { return (x + 63) / 64 * 64; }
size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

// Trailing columns whose digits are held at a time: at most 1 GB of them.  The more columns a
// launch takes, the fuller its last wave: 4096 x 4096, p = 16, f = 2, Rbar 8.9 -> 8.3 ms, update
// 11.3 -> 11.1 ms in place of 4096 columns at a time.
int64_t col_block(int64_t M, int64_t N) {
  const int64_t per = (int64_t)kD * up64(M) * 2;
  return std::min<int64_t>(N, std::max<int64_t>(512, ((int64_t)1 << 30) / per / 64 * 64));
}
constexpr int kMaxSplits = 8;

PFN_cuTensorMapEncodeTiled_v12000 encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

bool encode(CUtensorMap* tm, void* base, int64_t inner, int64_t outer, uint32_t box_rows) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = encoder();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)outer};
  cuuint64_t strides[1] = {(cuuint64_t)inner * 2};
  cuuint32_t box[2] = {BK, box_rows};
  cuuint32_t es[2] = {1, 1};
  return enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

struct F64Gemm {
  int64_t M, N, b, kpm, kpb, cols;  // kpm, kpb: plane strides along the rows and the panel width
  unsigned short *qc, *qr, *bt, *rb;
  int *eqc, *eqr, *ebt, *erb;
  int num_sms;
  CUtensorMap mqc, mqr, mbt, mrb;
};

// Workspace of the handle (0: its updates are too small to gain, or too tall, or the panel is wider
// than one sum of the update's K may be).
size_t f64_gemm_bytes(int64_t M, int64_t N, int64_t b) {
  if (M > (int64_t)kMaxSplits * kMaxK || b > kMaxK || !f64_gemm_pays(M, N - b, b)) return 0;
  const int64_t kpm = up64(M), kpb = up64(b), cols = col_block(M, N);
  return al256((size_t)b * kD * kpm * 2) + al256((size_t)M * kD * kpb * 2) +
         al256((size_t)cols * kD * kpm * 2) + al256((size_t)cols * kD * kpb * 2) +
         al256((size_t)(b + M + 2 * cols) * 4);
}

F64Gemm* f64_gemm_create(int64_t M, int64_t N, int64_t b, void* ws, int num_sms) {
  F64Gemm* t = new (std::nothrow) F64Gemm();
  if (!t) return nullptr;
  t->M = M;
  t->N = N;
  t->b = b;
  t->kpm = up64(M);
  t->kpb = up64(b);
  t->cols = col_block(M, N);
  t->num_sms = num_sms;
  char* p = static_cast<char*>(ws);
  auto take = [&](size_t bytes) { char* r = p; p += al256(bytes); return r; };
  t->qc = reinterpret_cast<unsigned short*>(take((size_t)b * kD * t->kpm * 2));
  t->qr = reinterpret_cast<unsigned short*>(take((size_t)M * kD * t->kpb * 2));
  t->bt = reinterpret_cast<unsigned short*>(take((size_t)t->cols * kD * t->kpm * 2));
  t->rb = reinterpret_cast<unsigned short*>(take((size_t)t->cols * kD * t->kpb * 2));
  t->eqc = reinterpret_cast<int*>(p);
  t->eqr = t->eqc + b;
  t->ebt = t->eqr + M;
  t->erb = t->ebt + t->cols;
  if (!encode(&t->mqc, t->qc, kD * t->kpm, b, BM) || !encode(&t->mqr, t->qr, kD * t->kpb, M, BM) ||
      !encode(&t->mbt, t->bt, kD * t->kpm, t->cols, BN) ||
      !encode(&t->mrb, t->rb, kD * t->kpb, t->cols, BN)) {
    delete t;
    return nullptr;
  }
  return t;
}

void f64_gemm_destroy(F64Gemm* t) { delete t; }

// Digits of the panel Qbar (M x bk at Q, ld ldq) for both products.
cudaError_t f64_gemm_panel(F64Gemm* t, const double* Q, int64_t ldq, int bk, cudaStream_t st) {
  k_f64_digits_cols<<<bk, 256, 0, st>>>(Q, ldq, t->M, t->kpm, t->kpm, t->qc, t->eqc);
  k_f64_digits_rows<<<(unsigned)((t->M + 31) / 32), 256, 0, st>>>(Q, ldq, t->M, bk, (int)up64(bk),
                                                                  t->kpb, t->qr, t->eqr);
  return cudaGetLastError();
}

int64_t f64_gemm_cols(const F64Gemm* t) { return t->cols; }

namespace {
cudaError_t launch_oz(const CUtensorMap& a, const CUtensorMap& b, const OzJob& job, int num_sms,
                      cudaStream_t st) {
  if (job.kchunk > kMaxK) return cudaErrorInvalidValue;  // the sums would overflow
  cudaError_t e = cudaFuncSetAttribute((const void*)k_f64_gemm,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemTotal);
  if (e != cudaSuccess) return e;
  const int units = job.m_tiles * job.n_tiles * job.splits;
  k_f64_gemm<<<std::min(units, num_sms), kThreads, kSmemTotal, st>>>(a, b, job);
  return cudaGetLastError();
}
}  // namespace

// Partials P[s] (bk x w, ld bk) of Qbar^T B, B (M x w, ld ldb), w <= f64_gemm_cols; *splits
// receives their number (at most 8).
cudaError_t f64_gemm_rbar(F64Gemm* t, const double* B, int64_t ldb, int64_t w, int bk, double* P,
                          int* splits, int* status, cudaStream_t st) {
  k_f64_digits_cols<<<(unsigned)w, 256, 0, st>>>(B, ldb, t->M, t->kpm, t->kpm, t->bt, t->ebt);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  OzJob job{};
  job.epi = 0;
  job.m_tiles = (bk + BM - 1) / BM;
  job.n_tiles = (int)((w + BN - 1) / BN);
  job.K = t->kpm;
  // the split whose launch finishes first: waves times stages of a unit, a reading of the
  // accumulators counted as one stage of a chunk more
  const int64_t kb = t->kpm / BK, tiles = (int64_t)job.m_tiles * job.n_tiles;
  double best = -1.0;
  for (int s = (int)((kb * BK + kMaxK - 1) / kMaxK); s <= kMaxSplits; ++s) {
    const int64_t kc = ((kb + s - 1) / s + kChunk - 1) / kChunk * kChunk;
    if (kc * BK > kMaxK) continue;
    const int64_t units = tiles * ((kb + kc - 1) / kc);
    const double cost = (double)((units + t->num_sms - 1) / t->num_sms) * (double)(kc + 2) * (1.0 + 0.02 * s);
    if (best < 0.0 || cost < best) {
      best = cost;
      job.kchunk = kc * BK;
    }
  }
  if (best < 0.0) return cudaErrorInvalidValue;
  job.splits = (int)((t->kpm + job.kchunk - 1) / job.kchunk);
  *splits = job.splits;
  job.kp_a = (int)t->kpm;
  job.kp_b = (int)t->kpm;
  job.mrows = bk;
  job.ncols = w;
  job.ea = t->eqc;
  job.eb = t->ebt;
  job.out = P;
  job.ldo = bk;
  job.split_stride = (int64_t)bk * w;
  job.status = status;
  return launch_oz(t->mqc, t->mbt, job, t->num_sms, st);
}

// C (M x w, ld ldc) -= Qbar Rb, Rb (bk x w, ld bk), w <= f64_gemm_cols.
cudaError_t f64_gemm_update(F64Gemm* t, const double* Rb, int64_t w, int bk, double* C, int64_t ldc,
                            int* status, cudaStream_t st) {
  const int64_t kend = up64(bk);
  k_f64_digits_cols<<<(unsigned)w, 256, 0, st>>>(Rb, bk, bk, kend, t->kpb, t->rb, t->erb);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  OzJob job{};
  job.epi = 1;
  job.m_tiles = (int)((t->M + BM - 1) / BM);
  job.n_tiles = (int)((w + BN - 1) / BN);
  job.splits = 1;
  job.K = kend;
  job.kchunk = kend;
  job.kp_a = (int)t->kpb;
  job.kp_b = (int)t->kpb;
  job.mrows = t->M;
  job.ncols = w;
  job.ea = t->eqr;
  job.eb = t->erb;
  job.out = C;
  job.ldo = ldc;
  job.status = status;
  return launch_oz(t->mqr, t->mrb, job, t->num_sms, st);
}

cudaError_t bounds_take_f64_gemm(int* code, int* site) { return bounds_take_here(code, site); }

}  // namespace cqr
