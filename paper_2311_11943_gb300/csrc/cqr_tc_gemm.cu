// cqr_tc_gemm.cu -- tensor-core trailing update of PBMGS for FP32 storage (sm_103a):
//   GEMM1  Rbar = Qbar^T Q[:, j0:j0+w]        (M_mma = panel columns, K = all M rows, split-K)
//   GEMM2  Q[:, j0:j0+w] -= Qbar Rbar          (M_mma = rows, K = panel width)
// (Appendix A, Algorithm PBMGS, the All-reduce product and the trailing update.)
//
// One persistent, warp-specialised kernel computes D = sum_p A_p B_p^T for up to three
// (A_p, B_p) operand pairs, every operand K-major, with tcgen05.mma kind::tf32 or kind::f16
// (M = 128, N = 128, 32 bytes of K per instruction) accumulating in tensor memory (TMEM, FP32):
//   warp 0      TMA producer: cp.async.bulk.tensor tiles (128-byte swizzle) into a ring of
//               shared-memory stages, completion counted on an mbarrier per stage
//   warp 1      allocates TMEM; one thread issues the MMAs and tcgen05.commit's each stage
//               back to the producer and each finished tile to the epilogue
//   warps 2-3   (and 12-13) split the streamed FP32 B tile in shared memory into its hi tile (in
//               place) and lo tile (the buffer behind it)
//   warps 4-11  epilogue, two warps per quarter of the TMEM lanes: tcgen05.ld 32 lanes x 32
//               columns per warp (alternate column chunks), then either store the FP32
//               partial (GEMM1) or subtract it from Q in place (GEMM2)
// A work unit is one 128 x 128 output tile, or, for GEMM1 in 3xTF32 with a 256-column panel,
// the two vertically adjacent tiles of one B tile (two accumulators; B is loaded and split
// once for both).
// The mode CQR_MMA_3XTF32 forms hi*hi + hi*lo + lo*hi of operands split into two 11-bit halves
// and so recovers about FP32 accuracy.  The halves are FP16, which has TF32's 11 bits in half the
// bytes and at twice the rate; what FP16 lacks, TF32's exponent range, comes from a power of two
// per column (exact to apply and to take out): orthonormal columns are multiplied by 2^12,
// trailing columns and those of Rbar by the power that takes their largest magnitude into [2^13,
// 2^14), the columns of a panel by that which takes their norm into [2^9, 2^10) when its block pass
// begins.  An entry keeps its 22 bits down to 2^-16 of the column's largest, and is off by at most
// 2^-38 of it below.  The magnitudes of the trailing columns are taken by the update that writes
// them, so what is left of a column whose large part was taken out keeps its digits, and a
// column that grows (a panel far from orthogonal) does not overflow.  Measured
// against 64 bits: R of 8192 x 8192 1.4e-5 -> 7.7e-6, of 16384 x 2048 6.9e-6 -> 3.7e-6 relative to
// TF32 halves (fewer roundings in the accumulators).  8192 x 8192, p = 16, b = 256, all panels:
// Rbar 5.0 -> 2.95 ms, block pass 8.1 -> 5.4 ms, update 4.94 -> 4.38 ms, 3.52 ms with C
// through shared memory (CT below; one pass over the trailing columns is 1.6 ms at the copy
// rate) and 3.69 ms with the columns' magnitudes.
// The small operands (panel and Rbar) are split into hi/lo planes in global memory by helper
// kernels.
// Every mbarrier wait is bounded: on expiry the kernel records CQR_ETIMEOUT, stops issuing,
// waits (bounded) for its own copies, frees TMEM and returns.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <new>

#include "coded_qr.h"
#include "cqr_device.cuh"
#include "cqr_tc_gemm.cuh"
#include "cqr_umma.cuh"

namespace cqr {

namespace {

using namespace umma;

constexpr int BM = 128;       // UMMA M (TMEM lanes)
constexpr int BN = 128;       // UMMA N (TMEM columns)
// TMEM columns: two accumulator buffers of U 128 x 128 accumulators (a power of two, <= 512)
template <int U>
constexpr int tmem_cols() { return 2 * U * BN; }
constexpr int kEpiWarps = 8;  // two per TMEM lane quarter, each draining half the columns
constexpr int kMaxSplits = 16;
// C ring of an epilogue warp (CT): chunks of 32 rows x 32 columns, 4 KB
constexpr int kCSlots = 3;
constexpr uint32_t kCBytes = 32 * 32 * 4;
constexpr uint32_t kTileBytesA = BM * 128;  // 16 KB: 128 rows of one 128-byte swizzle row
constexpr uint32_t kTileBytesB = BN * 128;  // 16 KB

// Operand type of the MMAs: TF32 (kind::tf32), BF16 or FP16 (kind::f16, A and B of the same
// type).  One stage of K is one 128-byte swizzle row of the operand type, 32 TF32 or 64 16-bit
// elements; each tcgen05.mma consumes 32 bytes of it (8 TF32 or 16 16-bit elements).
enum Kind { kTF32 = 0, kBF16 = 1, kF16 = 2 };
template <int KD>
struct Op {
  static constexpr int KE = KD == kTF32 ? 32 : 64;
  static constexpr int UK = KD == kTF32 ? 8 : 16;
};

// Warps 2 and 3 split the raw B tile.  FP16 adds two more after the epilogue's (one row of the
// tile per thread), since a stage's products take half as long per element as in TF32; launches
// without a split keep the registers for the epilogue instead.
template <int KD, bool SB>
struct Warps {
  static constexpr int kSplit = KD == kF16 && SB ? 4 : 2;
  static constexpr int kThreads = 32 * (2 + kSplit + kEpiWarps);
};

// Instruction descriptor: D FP32, both operands K-major, N and M encoded; A/B format FP16 (0),
// BF16 (1) or TF32 (2).
template <int KD>
constexpr uint32_t idesc() {
  constexpr uint32_t fmt = KD == kTF32 ? 2u : KD == kBF16 ? 1u : 0u;
  return (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(BN >> 3) << 17) |
         ((uint32_t)(BM >> 4) << 24);
}

template <int KD>
__device__ __forceinline__ void mma_op(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t accum) {
  if (KD != kTF32)
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(a), "l"(b), "r"(idesc<KD>()), "r"(accum)
        : "memory");
  else
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(a), "l"(b), "r"(idesc<KD>()), "r"(accum)
        : "memory");
}

// The FP16 scale of a column from the bits of its largest magnitude: the power of two that takes it
// into [2^13, 2^14), 1 for a column that is zero or not finite.
__device__ __forceinline__ float f16_scale(unsigned m) {
  const int e = (int)(m >> 23);
  if (m == 0u || e == 255) return 1.f;
  return __int_as_float(min(253, 267 - max(e, 1)) << 23);
}
// 1 / s of a power of two s within 2^-126 .. 2^126
__device__ __forceinline__ float pow2_inv(float s) { return __int_as_float((254 << 23) - __float_as_int(s)); }

__device__ __forceinline__ float tf32_hi(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

// ------------------------------------------------------------------ the GEMM kernel
struct TcMaps {
  CUtensorMap a[2];  // A hi / lo (lo unused for one product)
  CUtensorMap b[2];  // B hi / lo; with an in-smem split only b[0] (raw FP32) is loaded
  CUtensorMap c;     // subtract epilogue: the FP32 output (Q), boxes of 32 rows x BN columns
};

struct TcJob {
  int nprod;          // 1 (TF32) or 3 (3xTF32)
  int epi;            // 0: store partial P[s] ; 1: C -= D
  int prefetch_c;     // epi 1: prefetch each output tile into L2 when its loads start
  int pair_n;         // B from planes: work units of two N tiles when n_tiles is even
  int64_t c_col0;     // epi 1: column of `out` in the tensor map of C
  int m_tiles, n_tiles, splits;
  int64_t a_row0;     // A tile y coordinate offset (rows of the MMA M dimension)
  int64_t b_row0;     // B tile y coordinate offset
  int64_t k0;         // K start
  int64_t kchunk;     // K per split (multiple of the stage K)
  int64_t K;          // K end (exclusive)
  int64_t mrows;      // valid D rows (M dimension)
  int64_t ncols;      // valid D columns (N dimension)
  float* out;         // epi 0: P base; epi 1: C base (already offset to column j0)
  int64_t ldo;        // leading dimension of out
  int64_t split_stride;  // epi 0: elements between split partials
  // FP16 operands: raw B rows are multiplied by the scale of bmax (nullptr: bconst) before the
  // split, the epilogue of C -= D multiplies D by oconst and, column by column, by oinv (nullptr:
  // 1), and with CT leaves the largest magnitudes of the new columns in cmax
  const unsigned* bmax;
  const float* oinv;
  unsigned* cmax;
  float bconst, oconst;
  int* status;
};

template <int STAGES, int NA, int NB, int MP = 1, int NP = 1, bool CT = false>
struct Smem {
  // per stage: NA A tiles for each of the MP M tiles, then NB B tiles for each of the NP N
  // tiles (each 1024-byte aligned, 16 KB)
  static constexpr uint32_t kStageBytes = MP * NA * kTileBytesA + NP * NB * kTileBytesB;
  static constexpr uint32_t kTiles = STAGES * kStageBytes;
  static constexpr uint32_t kRing = CT ? kEpiWarps * kCSlots * kCBytes : 0;
  static constexpr uint32_t kTotal = kTiles + kRing + 1024 /*alignment*/ + 512 /*barriers*/;
  // full/ready/empty per stage, acc_full[2], acc_empty[2], C ring, TMEM slot, abort flag
  static_assert(STAGES * 3 * 8 + 4 * 8 + kEpiWarps * kCSlots * 8 + 8 <= 512, "barrier region too small");
  static_assert(kTotal <= 227 * 1024, "shared memory");
};

// Programmatic dependent launch: a kernel launched with programmatic stream serialization may
// start while its predecessor in the stream finishes.  Every kernel here waits for the
// predecessor's completion (and memory) before touching any data, and only then lets its own
// successor launch, so at most one kernel ahead is resident and waiting.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// MP = 2: a work unit is a pair of vertically adjacent M tiles on the same N tile (m_tiles
// even): the B tile is loaded (and split) once for both, and two accumulators are formed.
// NP = 2: a pair of adjacent N tiles on the same M tile (n_tiles even, B from planes): the A
// tiles are loaded once for both.  MP NP <= 2.
// SB: B arrives as raw FP32 and is split in shared memory.
// CT: C -= D with C through shared memory: each epilogue warp streams its chunks of C by TMA, two
// ahead of the one at work, and stores them by TMA.  With loads to registers a warp had one chunk
// in flight and only between its accumulator and its stores: 4096 x 4096, b = 128, 1.34 -> 1.05 ms
// for all panels, 8192 x 8192, b = 256, 4.38 -> 3.52 ms, although the ring leaves two operand
// stages in place of three.
template <int KD, bool SB, int STAGES, int NA, int NB, int MP, int NP, bool CT>
__global__ void __launch_bounds__(Warps<KD, SB>::kThreads, 1) k_tc_gemm(const __grid_constant__ TcMaps maps,
                                                          const TcJob job) {
  static_assert(MP * NP <= 2 && (!SB || NP == 1), "at most two accumulators per buffer");
  static_assert(!CT || (MP * NP == 1 && !SB && kEpiWarps == 8), "two chunks of each tile per epilogue warp");
  using S = Smem<STAGES, NA, NB, MP, NP, CT>;
  constexpr int kAcc = MP * NP;  // accumulators per work unit
  constexpr int kTmemCols = tmem_cols<kAcc>();
  constexpr bool BF = KD != kTF32;  // 16-bit operands
  constexpr int BK = Op<KD>::KE;
  constexpr int UMMA_K = Op<KD>::UK;
  extern __shared__ __align__(1024) unsigned char smraw[];
  const uint32_t base_u = su32(smraw);
  const uint32_t tiles_u = (base_u + 1023u) & ~1023u;
  unsigned char* tiles = smraw + (tiles_u - base_u);
  uint64_t* full = reinterpret_cast<uint64_t*>(tiles + S::kTiles + S::kRing);
  uint64_t* ready = full + STAGES;     // B split done (3xTF32 in-smem split)
  uint64_t* empty = ready + STAGES;
  uint64_t* acc_full = empty + STAGES;  // [2]: one per TMEM accumulator buffer
  uint64_t* acc_empty = acc_full + 2;   // [2]
  uint64_t* cfull = acc_empty + 2;      // [kEpiWarps][kCSlots] (CT)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(cfull + kEpiWarps * kCSlots);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // the output tiles stay inside `out` (uniform over the launch: before any barrier or TMEM
  // allocation)
  CQR_CHECK(job.ldo >= job.mrows && (int64_t)job.m_tiles * BM >= job.mrows &&
                (int64_t)job.n_tiles * BN >= job.ncols && job.m_tiles % MP == 0 &&
                job.n_tiles % NP == 0 && (NP == 1 || !SB), 401);
  const int mu = job.m_tiles / MP;  // work units along M
  const int total_tiles = mu * (job.n_tiles / NP) * job.splits;
  const int nkb_full = (int)(job.kchunk / BK);

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&ready[s], 32 * Warps<KD, SB>::kSplit);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], kEpiWarps);
    }
    if (CT)
      for (int i = 0; i < kEpiWarps * kCSlots; ++i) mbar_init(&cfull[i], 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    prefetch_tmap(&maps.a[0]);
    prefetch_tmap(&maps.b[0]);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     su32(tmem_slot)),
                 "r"((uint32_t)kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_wait();
  pdl_trigger();

  // K blocks of tile t
  auto kblocks = [&](int split) -> int {
    const int64_t k0 = job.k0 + (int64_t)split * job.kchunk;
    int64_t k1 = k0 + job.kchunk;
    if (k1 > job.K) k1 = job.K;
    const int64_t n = k1 > k0 ? (k1 - k0 + BK - 1) / BK : 0;
    return (int)(n < nkb_full ? n : nkb_full);
  };

  if (warp == 0) {
    if (lane == 0) {
      int it = 0;
      for (int t = blockIdx.x; t < total_tiles && !*abort_flag; t += gridDim.x) {
        const int split = t % job.splits;
        const int mn = t / job.splits;
        const int mt = (mn % mu) * MP, nt = (mn / mu) * NP;  // first M and N tiles of the unit
        const int nk = kblocks(split);
        const int64_t kbase = job.k0 + (int64_t)split * job.kchunk;
        if (job.prefetch_c) {
          // the output tiles (BM rows x BN columns of C) are read by the epilogue once this
          // unit's products are done: start bringing them into L2 now
          for (int n = 0; n < NP; ++n) {
            const int y = (int)(job.c_col0 + (int64_t)(nt + n) * BN);
            for (int r = 0; r < BM; r += 32) tma_prefetch_l2(&maps.c, mt * BM + r, y);
          }
        }
        for (int kb = 0; kb < nk; ++kb, ++it) {
          const int s = it % STAGES;
          if (!mbar_wait(&empty[s], ((it / STAGES) & 1) ^ 1, abort_flag)) break;
          const uint32_t st = tiles_u + s * S::kStageBytes;
          const int x = (int)(kbase + (int64_t)kb * BK);
          const int ya = (int)(job.a_row0 + (int64_t)mt * BM);
          const int yb = (int)(job.b_row0 + (int64_t)nt * BN);
          // raw FP32 B for the in-smem split: one 32-element box (TF32) or two (BF16: 64
          // elements of K, split in place into the BF16 hi and lo tiles)
          const int nb_load = SB ? (BF ? 2 : 1) : NB;
          mbar_expect_tx(&full[s], MP * NA * kTileBytesA + NP * nb_load * kTileBytesB);
#pragma unroll
          for (int m = 0; m < MP; ++m)
            for (int p = 0; p < NA; ++p)
              tma_load_2d(st + (m * NA + p) * kTileBytesA, &maps.a[p], x, ya + m * BM, &full[s]);
#pragma unroll
          for (int n = 0; n < NP; ++n)
            for (int p = 0; p < nb_load; ++p) {
              const bool raw = SB;
              tma_load_2d(st + MP * NA * kTileBytesA + (n * NB + p) * kTileBytesB,
                          raw ? &maps.b[0] : &maps.b[p], raw ? x + 32 * p : x, yb + n * BN,
                          &full[s]);
            }
        }
      }
      // the last load issued into each stage has landed before the CTA may exit (bounded)
      for (int i = (it > STAGES ? it - STAGES : 0); i < it; ++i) {
        const long long t0 = clock64();
        while (!mbar_test(&full[i % STAGES], (i / STAGES) & 1) && clock64() - t0 < kWaitLimitCycles) {
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      int it = 0, tl = 0;
      for (int t = blockIdx.x; t < total_tiles && !*abort_flag; t += gridDim.x, ++tl) {
        const int split = t % job.splits;
        const int nk = kblocks(split);
        // two accumulator buffers: the epilogue drains unit tl-1 while unit tl accumulates;
        // a buffer holds MP accumulators of BN columns
        const int buf = tl & 1;
        const uint32_t acc = tmem + (uint32_t)(buf * kAcc * BN);
        if (!mbar_wait(&acc_empty[buf], ((tl >> 1) & 1) ^ 1, abort_flag)) break;
        tc_fence_after();
        bool ok = true;
        for (int kb = 0; kb < nk; ++kb, ++it) {
          const int s = it % STAGES;
          uint64_t* gate = SB ? &ready[s] : &full[s];
          if (!mbar_wait(gate, (it / STAGES) & 1, abort_flag)) { ok = false; break; }
          tc_fence_after();
          const uint32_t st = tiles_u + s * S::kStageBytes;
#pragma unroll
          for (int ks = 0; ks < BK / UMMA_K; ++ks) {
            const uint32_t off = ks * 32;  // 32 bytes of K per instruction
            const uint32_t acc0 = (kb > 0 || ks > 0) ? 1u : 0u;
#pragma unroll
            for (int m = 0; m < MP; ++m)
#pragma unroll
              for (int n = 0; n < NP; ++n) {
                const uint32_t am = acc + (uint32_t)((m * NP + n) * BN);
                const uint32_t a_hi = st + m * NA * kTileBytesA, a_lo = a_hi + kTileBytesA;
                const uint32_t b_hi = st + MP * NA * kTileBytesA + n * NB * kTileBytesB;
                const uint32_t b_lo = b_hi + kTileBytesB;
                mma_op<KD>(am, sdesc(a_hi + off), sdesc(b_hi + off), acc0);
                if (job.nprod == 3) {
                  mma_op<KD>(am, sdesc(a_hi + off), sdesc(b_lo + off), 1u);
                  mma_op<KD>(am, sdesc(a_lo + off), sdesc(b_hi + off), 1u);
                }
              }
          }
          mma_commit(&empty[s]);
        }
        if (!ok) break;
        mma_commit(&acc_full[buf]);
      }
    }
  } else if (warp < 4 || warp >= 4 + kEpiWarps) {
    if constexpr (SB) {
      const int tt = threadIdx.x - (warp < 4 ? 64 : 32 * (2 + kEpiWarps));
      int it = 0;
      for (int t = blockIdx.x; t < total_tiles && !*abort_flag; t += gridDim.x) {
        const int split = t % job.splits;
        const int nk = kblocks(split);
        float sc = job.bconst;  // FP16: the scale of this thread's row of the B tile
        if (KD == kF16 && job.bmax) {
          const int64_t j = (int64_t)(t / job.splits / mu) * NP * BN + tt;
          sc = j < job.ncols ? f16_scale(job.bmax[j]) : 1.f;
        }
        bool ok = true;
        for (int kb = 0; kb < nk; ++kb, ++it) {
          const int s = it % STAGES;
          if (!mbar_wait(&full[s], (it / STAGES) & 1, abort_flag)) { ok = false; break; }
          float4* raw = reinterpret_cast<float4*>(tiles + s * S::kStageBytes + MP * NA * kTileBytesA);
          float4* lo = raw + kTileBytesB / 16;
          if (!BF) {
            for (int e = tt; e < (int)(kTileBytesB / 16); e += 64) {
              const float4 x = raw[e];
              float4 h, l;
              h.x = tf32_hi(x.x); l.x = x.x - h.x;
              h.y = tf32_hi(x.y); l.y = x.y - h.y;
              h.z = tf32_hi(x.z); l.z = x.z - h.z;
              h.w = tf32_hi(x.w); l.w = x.w - h.w;
              raw[e] = h;
              lo[e] = l;
            }
          } else {
            // row r of the two raw FP32 tiles (K 0..31 and 32..63, 16-byte chunks swizzled by
            // r % 8) becomes row r of the BF16 hi tile (first 16 KB) and lo tile (second):
            // a thread reads both raw rows before writing, and no other thread touches row r
            for (int r = tt; r < BN; r += 32 * Warps<KD, SB>::kSplit) {
              float v[64];
#pragma unroll
              for (int c = 0; c < 16; ++c) {
                const int tile = c >> 3, lc = c & 7;
                const float4 x = raw[tile * (kTileBytesB / 16) + r * 8 + (lc ^ (r & 7))];
                v[4 * c] = x.x; v[4 * c + 1] = x.y; v[4 * c + 2] = x.z; v[4 * c + 3] = x.w;
              }
#pragma unroll
              for (int c = 0; c < 8; ++c) {
                uint32_t hw[4], lw[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                  const float a0 = v[8 * c + 2 * q], a1 = v[8 * c + 2 * q + 1];
                  if constexpr (KD == kF16) {
                    const float x0 = a0 * sc, x1 = a1 * sc;
                    const __half2 h = __floats2half2_rn(x0, x1);
                    const float2 f = __half22float2(h);
                    const __half2 l = __floats2half2_rn(x0 - f.x, x1 - f.y);
                    memcpy(&hw[q], &h, 4);
                    memcpy(&lw[q], &l, 4);
                    continue;
                  }
                  const __nv_bfloat16 h0 = __float2bfloat16_rn(a0), h1 = __float2bfloat16_rn(a1);
                  const __nv_bfloat16 l0 = __float2bfloat16_rn(a0 - __bfloat162float(h0));
                  const __nv_bfloat16 l1 = __float2bfloat16_rn(a1 - __bfloat162float(h1));
                  hw[q] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
                  lw[q] = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
                }
                const int pc = r * 8 + (c ^ (r & 7));
                reinterpret_cast<uint4*>(raw)[pc] = make_uint4(hw[0], hw[1], hw[2], hw[3]);
                if (job.nprod == 3) reinterpret_cast<uint4*>(lo)[pc] = make_uint4(lw[0], lw[1], lw[2], lw[3]);
              }
            }
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          mbar_arrive(&ready[s]);
        }
        if (!ok) break;
      }
    }
  } else if constexpr (CT) {
    // chunk g of this warp: 32-column chunk half + 2 (g % 2) of the CTA's unit g / 2
    const int ew = warp & 3, half = (warp - 4) >> 2;
    const uint32_t ring_u = tiles_u + S::kTiles + (uint32_t)(warp - 4) * kCSlots * kCBytes;
    unsigned char* ring = tiles + S::kTiles + (size_t)(warp - 4) * kCSlots * kCBytes;
    uint64_t* cbar = cfull + (warp - 4) * kCSlots;
    uint32_t phase = 0, pending = 0;  // of each slot
    // the chunk's rows and columns; whole: it goes through the ring (all its columns belong to the
    // job; rows past M are dropped by the tensor map)
    auto place = [&](int g, int64_t& row0, int64_t& col0) {
      const int t = blockIdx.x + (g >> 1) * gridDim.x;
      if (t >= total_tiles) return false;
      row0 = (int64_t)(t % mu) * BM + ew * 32;
      col0 = (int64_t)(t / mu) * BN + (half + 2 * (g & 1)) * 32;
      return row0 < job.mrows && col0 + 32 <= job.ncols;
    };
    auto cload = [&](int g) {
      int64_t row0, col0;
      if (!place(g, row0, col0)) return;
      const int s = g % kCSlots;
      pending |= 1u << s;
      if (lane == 0) {
        mbar_expect_tx(&cbar[s], kCBytes);
        tma_load_2d(ring_u + s * kCBytes, &maps.c, (int)row0, (int)(job.c_col0 + col0), &cbar[s]);
      }
    };
    cload(0);
    cload(1);
    int tl = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < total_tiles && ok; t += gridDim.x, ++tl) {
      const int buf = tl & 1;
      ok = __all_sync(~0u, mbar_wait(&acc_full[buf], (tl >> 1) & 1, abort_flag) ? 1 : 0);
      if (!ok) break;
      tc_fence_after();
#pragma unroll 1
      for (int u = 0; u < 2; ++u) {
        const int g = 2 * tl + u, s = g % kCSlots, c = half + 2 * u;
        if (lane == 0) bulk_wait_read();  // the slot of chunk g + 2 was stored from by chunk g - 1
        __syncwarp();
        cload(g + 2);
        int64_t row0 = 0, col0 = 0;
        const bool whole = place(g, row0, col0);
        const int64_t row = row0 + lane;
        float inv = 1.f;
        if (job.oinv && col0 + lane < job.ncols) inv = job.oinv[col0 + lane];
        unsigned big = 0u, seen = ~0u;  // what the column has already: most chunks need no atomic
        if (col0 + lane < job.ncols) seen = *reinterpret_cast<volatile unsigned*>(job.cmax + col0 + lane);
        float v[32];
        tmem_ld32(tmem + ((uint32_t)(ew * 32) << 16) + (uint32_t)(buf * BN + c * 32), v);
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = v[i] * job.oconst * __shfl_sync(~0u, inv, i);
        if (whole) {
          ok = __all_sync(~0u, mbar_wait(&cbar[s], (phase >> s) & 1, abort_flag) ? 1 : 0);
          if (!ok) break;
          phase ^= 1u << s;
          pending &= ~(1u << s);
          // column i of the chunk is one 128-byte row of the box, its 16-byte units swizzled
          unsigned char* sl = ring + s * kCBytes + (lane & 3) * 4;
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            float* x = reinterpret_cast<float*>(sl + i * 128 + (((lane >> 2) ^ (i & 7)) << 4));
            *x -= v[i];
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) {
            tma_store_2d(&maps.c, (int)row0, (int)(job.c_col0 + col0), ring_u + s * kCBytes);
            bulk_commit();
          }
          // column `lane` of the chunk again, along its row of the box (no bank conflicts): 32 reads
          // across the lanes by __reduce_max_sync cost as much as a tenth of the launch
          const float4* y = reinterpret_cast<const float4*>(ring + s * kCBytes + lane * 128);
          float m = 0.f;
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const float4 c4 = y[k ^ (lane & 7)];
            m = fmaxf(fmaxf(m, fmaxf(fabsf(c4.x), fabsf(c4.y))), fmaxf(fabsf(c4.z), fabsf(c4.w)));
          }
          big = __float_as_uint(m);
        } else {
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            float c = 0.f;
            if (row < job.mrows && col0 + i < job.ncols) {
              float* x = job.out + row + (col0 + i) * job.ldo;
              c = *x - v[i];
              *x = c;
            }
            const unsigned m = __reduce_max_sync(~0u, __float_as_uint(c) & 0x7fffffffu);
            if (lane == i) big = m;
          }
        }
        if (big > seen) atomicMax(job.cmax + col0 + lane, big);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[buf]);
    }
    // nothing of this warp is in flight when the CTA exits (loads: bounded)
    for (int s = 0; s < kCSlots; ++s)
      if (pending >> s & 1) {
        const long long t0 = clock64();
        while (!mbar_test(&cbar[s], (phase >> s) & 1) && clock64() - t0 < kWaitLimitCycles) {
        }
      }
    if (lane == 0) bulk_wait();
  } else {
    // epilogue warps 4 .. 4+kEpiWarps-1: TMEM lanes 32 (warp % 4) .. +32 (a warp may only
    // read its own quarter of the lanes); the two warps of a quarter take alternate 32-column
    // chunks (of each of the unit's MP accumulators), so twice as many loads of the output
    // tile are in flight
    const int ew = warp & 3;
    const int half = (warp - 4) >> 2;
    constexpr int kChunks = BN / 32;
    int tl = 0;
    for (int t = blockIdx.x; t < total_tiles && !*abort_flag; t += gridDim.x, ++tl) {
      const int split = t % job.splits;
      const int mn = t / job.splits;
      const int mt = (mn % mu) * MP, nt = (mn / mu) * NP;
      const int buf = tl & 1;
      if (!mbar_wait(&acc_full[buf], (tl >> 1) & 1, abort_flag)) break;
      tc_fence_after();
      const bool has_k = kblocks(split) > 0;
#pragma unroll 1
      for (int q = half; q < kAcc * kChunks; q += kEpiWarps / 4) {
        const int a = q / kChunks, c = q % kChunks;  // accumulator a = m NP + n
        const int m = a / NP, n = a % NP;
        const int64_t row = (int64_t)(mt + m) * BM + ew * 32 + lane;
        const bool row_ok = row < job.mrows;
        float v[32];
        tmem_ld32(tmem + ((uint32_t)(ew * 32) << 16) + (uint32_t)((buf * kAcc + a) * BN + c * 32), v);
        if (!has_k)
#pragma unroll
          for (int i = 0; i < 32; ++i) v[i] = 0.f;
        const int64_t col0 = (int64_t)(nt + n) * BN + c * 32;
        if (job.epi == 0 || (KD == kF16 && SB)) {
          float* o = job.out + (int64_t)split * job.split_stride;
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const int64_t col = col0 + i;
            if (row_ok && col < job.ncols) o[row + col * job.ldo] = v[i];
          }
        } else {
          // the columns' factors, one per lane, before the loads of the output tile
          float inv = 1.f;
          if (KD == kF16 && job.oinv && col0 + lane < job.ncols) inv = job.oinv[col0 + lane];
          float old[32];
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const int64_t col = col0 + i;
            old[i] = (row_ok && col < job.ncols) ? job.out[row + col * job.ldo] : 0.f;
          }
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const int64_t col = col0 + i;
            if (KD == kF16) v[i] = v[i] * job.oconst * __shfl_sync(~0u, inv, i);
            if (row_ok && col < job.ncols) job.out[row + col * job.ldo] = old[i] - v[i];
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[buf]);
    }
  }

  __syncthreads();
  if (*abort_flag && threadIdx.x == 0) set_status(job.status, CQR_ETIMEOUT, 20);
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"((uint32_t)kTmemCols)
                 : "memory");
  }
}

// ------------------------------------------------------------------ helper kernels
// Panel split: Qbar = Q[:, kb : kb+bk] (M x bk) -> for GEMM1's A (column-major, ld ldk):
// Ak_hi / Ak_lo; for GEMM2's A (row-major, row stride bkp): At_hi / At_lo; columns k >= bk
// zero-filled up to bkp (and up to 128 columns for GEMM1's M tile).  With Qr != nullptr the
// finished panel is also copied into the row-major planes of all computed columns
// (Qr[r * ldrow + kb + k]), the K-major operand of the block reorthogonalisation; columns
// bk .. qcols - 1 of that copy are zero: a later product reads whole stages of K, the columns behind
// the last computed one against zero rows, and what an earlier factorisation left there need
// not be finite.
// Operand planes: x = hi + lo with hi = rna_tf32(x) (TF32; hi = x with one product, the MMA
// reads TF32 from the FP32 word) or hi = rn(x), lo = rn(x - hi) in BF16 or FP16 (there x is
// scaled: by cscale[k] where given, else by scale).
__device__ __forceinline__ void hilo(float x, int nplanes, float& h, float& l) {
  h = nplanes == 2 ? tf32_hi(x) : x;
  l = x - h;
}
__device__ __forceinline__ void hilo(float x, int, __half& h, __half& l) {
  h = __float2half_rn(x);
  l = __float2half_rn(x - __half2float(h));
}
__device__ __forceinline__ void hilo(float x, int, __nv_bfloat16& h, __nv_bfloat16& l) {
  h = __float2bfloat16_rn(x);
  l = __float2bfloat16_rn(x - __bfloat162float(h));
}

// One 32-row x 32-column tile per CTA: Q is read and Ak written along the rows (coalesced);
// the row-major planes (At, Qr) are written from a shared-memory transpose of the tile, so
// that consecutive threads write consecutive columns of a row.
template <typename P>
__global__ void __launch_bounds__(256) k_split_panel(const float* __restrict__ Q, int64_t ldq,
                                                     int64_t M, int bk, int bkp, int ak_cols,
                                                     int nplanes, P* __restrict__ Ak_hi,
                                                     P* __restrict__ Ak_lo, int64_t ldk,
                                                     P* __restrict__ At_hi, P* __restrict__ At_lo,
                                                     P* __restrict__ Qr_hi, P* __restrict__ Qr_lo,
                                                     int64_t ldrow, int64_t kb, int qcols, float scale,
                                                     const float* __restrict__ cscale) {
  __shared__ P sh[32][33], sl[32][33];
  pdl_wait();
  pdl_trigger();
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int64_t r0 = (int64_t)blockIdx.x * 32;
  const int k0 = blockIdx.y * 32;
  const int64_t r = r0 + tx;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int k = k0 + ty + 8 * i;
    const float x = (r < M && k < bk) ? Q[r + (int64_t)k * ldq] : 0.f;
    P h, l;
    hilo(x * (cscale && k < bk ? cscale[k] : scale), nplanes, h, l);
    if (r < M && k < ak_cols) {
      if (Ak_hi) Ak_hi[r + (int64_t)k * ldk] = h;
      if (Ak_lo && nplanes == 2) Ak_lo[r + (int64_t)k * ldk] = l;
    }
    sh[ty + 8 * i][tx] = h;
    sl[ty + 8 * i][tx] = l;
  }
  __syncthreads();
  const int k = k0 + tx;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t rr = r0 + ty + 8 * i;
    if (rr >= M) continue;
    const P h = sh[tx][ty + 8 * i], l = sl[tx][ty + 8 * i];
    if (At_hi && k < bkp) {
      At_hi[rr * bkp + k] = h;
      if (nplanes == 2) At_lo[rr * bkp + k] = l;
    }
    if (Qr_hi && k < qcols) {
      Qr_hi[rr * ldrow + kb + k] = h;
      if (nplanes == 2) Qr_lo[rr * ldrow + kb + k] = l;
    }
  }
}

// C -= sum_s P[s] in a fixed order of s (split-K partials of a C -= A B update; P[s] is
// mrows x ncols column-major with leading dimension mrows).
__global__ void k_tc_sub_partials(const float* __restrict__ P, int splits, int64_t mrows,
                                  int64_t ncols, float* __restrict__ C, int64_t ldc, float oconst,
                                  const float* __restrict__ oinv) {
  pdl_wait();
  pdl_trigger();
  const int64_t total = mrows * ncols;
  const int64_t stride = total;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = idx % mrows, c = idx / mrows;
    float s = 0.f;
    for (int sp = 0; sp < splits; ++sp) s += __ldcs(P + sp * stride + idx);
    C[r + c * ldc] -= oinv ? s * oconst * oinv[c] : s * oconst;
  }
}

// FP16 scales of `ncols` columns of C (M rows): cs[j] = the power of two that takes the 2-norm
// of column j into [2^9, 2^10), ci[j] = 1 / cs[j]; 1 for a column that is zero or not finite.
// One CTA per column; the largest magnitude first, so that the sum of squares cannot overflow
// or vanish (the second reading comes from the caches).
__global__ void __launch_bounds__(256) k_col_scale(const float* __restrict__ C, int64_t ldc, int64_t M,
                                                   float* __restrict__ cs, float* __restrict__ ci) {
  __shared__ float red[8];
  pdl_wait();
  pdl_trigger();
  const float* c = C + (int64_t)blockIdx.x * ldc;
  const int tid = threadIdx.x;
  float m = 0.f;
  for (int64_t r = tid; r < M; r += 256) m = fmaxf(m, fabsf(c[r]));
#pragma unroll
  for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(~0u, m, o));
  if ((tid & 31) == 0) red[tid >> 5] = m;
  __syncthreads();
  m = red[0];
#pragma unroll
  for (int w = 1; w < 8; ++w) m = fmaxf(m, red[w]);
  __syncthreads();
  int e = 0;
  const bool plain = m > 0.f && m <= 3.402823466e38f;
  if (plain) frexpf(m, &e);  // m in [2^(e-1), 2^e)
  // x 2^-e in two exact steps, so that neither factor leaves the range
  const float s1 = ldexpf(1.f, -(e / 2)), s2 = ldexpf(1.f, -(e - e / 2));
  float q = 0.f;
  for (int64_t r = tid; r < M; r += 256) {
    const float x = c[r] * s1 * s2;
    q += x * x;
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) q += __shfl_xor_sync(~0u, q, o);
  if ((tid & 31) == 0) red[tid >> 5] = q;
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < 8; ++w) q += red[w];
    float s = 1.f;
    if (plain && q <= 3.402823466e38f) {
      int eq;
      frexpf(sqrtf(q), &eq);  // the norm lies in [2^(e+eq-1), 2^(e+eq))
      s = ldexpf(1.f, min(126, max(-120, 10 - (e + eq))));
    }
    cs[blockIdx.x] = s;
    ci[blockIdx.x] = 1.f / s;
  }
}

// Row-major planes of the rectangle rows [r0, r0 + nr) x columns [c0, c0 + nc) from Q (after a
// recovery rebuilt those tiles): 32 x 32 tiles through shared memory, coalesced both ways.
template <typename P>
__global__ void __launch_bounds__(256) k_refresh_rect(const float* __restrict__ Q, int64_t ldq,
                                                      int64_t r0, int nr, int64_t c0, int nc,
                                                      int nplanes, P* __restrict__ Qr_hi,
                                                      P* __restrict__ Qr_lo, int64_t ldrow,
                                                      float scale) {
  __shared__ P sh[32][33], sl[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int rb = blockIdx.x * 32, cb = blockIdx.y * 32;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int r = rb + tx, c = cb + ty + 8 * u;
    P h, l;
    hilo((r < nr && c < nc) ? Q[r0 + r + (c0 + c) * ldq] * scale : 0.f, nplanes, h, l);
    sh[ty + 8 * u][tx] = h;
    sl[ty + 8 * u][tx] = l;
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int r = rb + ty + 8 * u, c = cb + tx;
    if (r >= nr || c >= nc) continue;
    Qr_hi[(r0 + r) * ldrow + c0 + c] = sh[tx][ty + 8 * u];
    if (nplanes == 2) Qr_lo[(r0 + r) * ldrow + c0 + c] = sl[tx][ty + 8 * u];
  }
}

// Block reorthogonalisation, reduce: the GEMM1 partials hold S^T = Qbar^T Q[:, 0:kb]
// (P[s][i + j bkp]); R[j, kb+i] += S[j][i] and S (column-major, ld ldrow, rows >= kb zero)
// goes into the B planes of the second product.  One 32 x 32 tile (i, j) per CTA: the
// partials are read along i and the sums go through shared memory, so R and S are written
// along j (both coalesced).
template <typename PT>
__global__ void __launch_bounds__(256) k_tc_reduce_t(const float* __restrict__ P, int splits,
                                                     int64_t split_stride, int64_t ldp, int bk,
                                                     int64_t kb, int64_t kbp, float* __restrict__ R,
                                                     int64_t ldr, int nplanes, PT* __restrict__ Sh,
                                                     PT* __restrict__ Sl, int64_t ldrow, float oconst,
                                                     const float* __restrict__ oinv) {
  __shared__ float tile[32][33];
  pdl_wait();
  pdl_trigger();
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int i0 = blockIdx.x * 32;
  const int64_t j0 = (int64_t)blockIdx.y * 32;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int i = i0 + tx;
    const int64_t j = j0 + ty + 8 * u;
    float s = 0.f;
    if (i < bk && j < kb)
      for (int sp = 0; sp < splits; ++sp) s += P[sp * split_stride + i + j * ldp];
    tile[ty + 8 * u][tx] = s * oconst;
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int i = i0 + ty + 8 * u;
    const int64_t j = j0 + tx;
    if (i >= bk || j >= kbp) continue;
    const float s = tile[tx][ty + 8 * u];
    if (j < kb) R[j + (kb + i) * ldr] += oinv ? s * oinv[i] : s;
    PT h, l;
    hilo(s, nplanes, h, l);
    Sh[j + i * ldrow] = h;
    if (nplanes == 2) Sl[j + i * ldrow] = l;
  }
}

// Split-K reduction of GEMM1: Rbar = sum_s P[s] (fixed order) into R (rows kb.., columns
// j0..) and into GEMM2's B operand planes (column-major, ld bkp, rows >= bk zero).
template <typename PT>
__global__ void k_tc_reduce(const float* __restrict__ P, int splits, int64_t split_stride, int64_t ldp,
                            int bk, int bkp, int64_t w, float* __restrict__ R, int64_t ldr,
                            int nplanes, PT* __restrict__ Bh, PT* __restrict__ Bl) {
  pdl_wait();
  pdl_trigger();
  const int64_t total = (int64_t)bkp * w;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = idx % bkp, j = idx / bkp;
    float s = 0.f;
    if (i < bk) {
      for (int sp = 0; sp < splits; ++sp) s += P[sp * split_stride + i + j * ldp];
      R[i + j * ldr] = s;
    }
    PT h, l;
    hilo(s, nplanes, h, l);
    Bh[idx] = h;
    if (nplanes == 2) Bl[idx] = l;
  }
}

// The same for FP16 operands, a warp per column: the partials hold Rbar times `qscale` and the scale
// of cmax[j], the planes Rbar times the scale of the column's own largest magnitude, whose
// inverse goes into ri[j]; cnext[j] is cleared for the update behind.
__global__ void __launch_bounds__(256) k_tc_reduce_f16(const float* __restrict__ P, int splits,
                                                       int64_t split_stride, int64_t ldp, int bk, int bkp,
                                                       int64_t w, float* __restrict__ R, int64_t ldr,
                                                       __half* __restrict__ Bh, __half* __restrict__ Bl,
                                                       float qinv, const unsigned* __restrict__ cmax,
                                                       float* __restrict__ ri, unsigned* __restrict__ cnext) {
  pdl_wait();
  pdl_trigger();
  constexpr int E = 4;  // entries of a lane in registers
  const int lane = threadIdx.x & 31;
  const int64_t j = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (j >= w) return;
  const float inv = pow2_inv(f16_scale(cmax[j]));
  const float* p = P + j * ldp;
  float* r = R + j * ldr;
  float v[E];
  unsigned m = 0u;
  for (int i0 = 0; i0 < bkp; i0 += 32 * E) {
#pragma unroll
    for (int u = 0; u < E; ++u) v[u] = 0.f;
    for (int sp = 0; sp < splits; sp += 8) {  // the loads of eight partials in flight, added in their order
      float x[8][E];
#pragma unroll
      for (int q = 0; q < 8; ++q)
#pragma unroll
        for (int u = 0; u < E; ++u) {
          const int i = i0 + 32 * u + lane;
          x[q][u] = i < bk && sp + q < splits ? p[(sp + q) * split_stride + i] : 0.f;
        }
#pragma unroll
      for (int q = 0; q < 8; ++q)
#pragma unroll
        for (int u = 0; u < E; ++u) v[u] += x[q][u];
    }
#pragma unroll
    for (int u = 0; u < E; ++u) {
      const int i = i0 + 32 * u + lane;
      v[u] = v[u] * qinv * inv;
      if (i < bk) r[i] = v[u];
      m = max(m, __float_as_uint(v[u]) & 0x7fffffffu);
    }
  }
  m = __reduce_max_sync(~0u, m);
  const float s = f16_scale(m);
  if (lane == 0) {
    ri[j] = pow2_inv(s);
    cnext[j] = 0u;
  }
  for (int i0 = 0; i0 < bkp; i0 += 32 * E) {
    if (bkp > 32 * E)  // written above by this lane
#pragma unroll
      for (int u = 0; u < E; ++u) {
        const int i = i0 + 32 * u + lane;
        v[u] = i < bk ? r[i] : 0.f;
      }
#pragma unroll
    for (int u = 0; u < E; ++u) {
      const int i = i0 + 32 * u + lane;
      if (i >= bkp) continue;
      __half h, l;
      hilo(v[u] * s, 2, h, l);
      Bh[i + j * bkp] = h;
      Bl[i + j * bkp] = l;
    }
  }
}

// Bits of the largest magnitude of every column of C (M rows), one CTA per column (a NaN counts as the
// largest).
__global__ void __launch_bounds__(256) k_col_max(const float* __restrict__ C, int64_t ldc, int64_t M,
                                                 unsigned* __restrict__ cmax) {
  __shared__ unsigned red[8];
  pdl_wait();
  pdl_trigger();
  const float* c = C + (int64_t)blockIdx.x * ldc;
  unsigned m = 0u;
#pragma unroll 4
  for (int64_t r = threadIdx.x; r < M; r += 256) m = max(m, __float_as_uint(c[r]) & 0x7fffffffu);
  m = __reduce_max_sync(~0u, m);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < 8; ++k) m = max(m, red[k]);
    cmax[blockIdx.x] = m;
  }
}

}  // namespace

// ------------------------------------------------------------------ host side
struct TcGemm {
  int mode;           // CQR_MMA_TF32 | _3XTF32 | _BF16 | _BF16X3
  int nplanes;        // 1 or 2
  int kind;           // operand type of the planes and the MMAs (Kind)
  int KE;             // K elements per stage (32 TF32, 64 16-bit)
  size_t pe;          // bytes per plane element
  int64_t M, N, b, bkp, ldq, ldk;
  float* Q;
  // panel operand planes, two buffers (panels of alternating parity), and the Rbar planes and
  // split-K partials of two update contexts (the look-ahead runs two updates concurrently)
  void *Ak_hi[2], *Ak_lo[2], *At_hi[2], *At_lo[2], *Bh[2], *Bl[2];
  float* P[2];
  void *Qr_hi, *Qr_lo, *Sh, *Sl;   // block reorthogonalisation operands
  // FP16: bits of the columns' largest magnitudes at a panel (by its parity) and the inverse scales
  // of the Rbar planes' columns; in the block pass, scales of the panel's columns and their inverses
  unsigned* cm[2];
  float *ri, *cs, *ci;
  int64_t n, ldrow;
  int num_sms;
  int* status;
  bool pdl = false;  // launches on pdl_st use programmatic dependent launch
  cudaStream_t pdl_st = nullptr;
  CUtensorMap tm_q_b;        // Q (FP32) as GEMM1's raw B (box 32 x BN)
  CUtensorMap tm_q_c;        // Q in chunks of 32 rows x 32 columns (CT)
  CUtensorMap tm_ak[2][2];   // [buffer][plane] panel, column-major (box KE x BM)
  CUtensorMap tm_at[2][2];   // [buffer][plane] panel, row-major (box KE x BM)
  CUtensorMap tm_bh[2][2];   // [context][plane] Rbar planes (box KE x BN)
  CUtensorMap tm_qr[2];      // computed columns, row-major (box KE x BM)
  CUtensorMap tm_s[2];       // S planes, column-major ld ldrow (box KE x BN)
};

namespace {

// The driver's tensor-map encoder, resolved through the runtime (the library does not link
// the driver library, so it loads on machines without a GPU driver).
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

bool encode_2d(CUtensorMap* tm, void* base, int kind, uint64_t inner, uint64_t outer,
               uint64_t row_bytes, uint32_t box_inner, uint32_t box_outer) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = encoder();
  if (!enc) return false;
  cuuint64_t dims[2] = {inner, outer};
  cuuint64_t strides[1] = {row_bytes};
  cuuint32_t box[2] = {box_inner, box_outer};
  cuuint32_t es[2] = {1, 1};
  CUresult r = enc(tm, kind == kTF32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                : kind == kBF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                                : CU_TENSOR_MAP_DATA_TYPE_FLOAT16,
                   2, base, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

// Kernel launch, with programmatic stream serialization when pdl is set.
template <typename... KArgs, typename... Args>
cudaError_t launch_k(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                     bool pdl, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = pdl ? at : nullptr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

template <int KD, bool SB, int STAGES, int NA, int NB, int MP = 1, int NP = 1, bool CT = false>
cudaError_t launch_gemm(const TcMaps& maps, const TcJob& job, int max_ctas, cudaStream_t st, bool pdl) {
  using S = Smem<STAGES, NA, NB, MP, NP, CT>;
  const void* fn = (const void*)k_tc_gemm<KD, SB, STAGES, NA, NB, MP, NP, CT>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::kTotal);
  if (e != cudaSuccess) return e;
  const int tiles = job.m_tiles / MP * (job.n_tiles / NP) * job.splits;
  const int grid = std::max(1, std::min(tiles, max_ctas));
  return launch_k(k_tc_gemm<KD, SB, STAGES, NA, NB, MP, NP, CT>, dim3(grid), dim3(Warps<KD, SB>::kThreads),
                  S::kTotal, st,
                  pdl, maps, job);
}

// GEMM1-shaped launches (B raw and split in shared memory, 3xTF32) take pairs of M tiles when
// the panel spans an even number of them (b = 256): the B tile is then loaded and split once
// for both halves of the panel, which halves the B traffic into shared memory per flop.
// CQR_GEMM_PAIR=0 keeps one M tile per work unit.
bool pair_m_tiles(const TcGemm* t, bool split, int m_tiles) {
  static const int env = [] {
    const char* e = getenv("CQR_GEMM_PAIR");
    return e ? atoi(e) : 1;
  }();
  return env != 0 && t->kind == kF16 && split && m_tiles % 2 == 0;
}

// Launches whose B comes from planes (GEMM2 and the block pass's second product) take pairs of
// N tiles when the job asks for it (TcJob::pair_n) and n_tiles is even: the A tiles are then
// loaded once for both: the block pass's second product (CQR_GEMM_NPAIR=0: never).
int npair_level() {
  static const int env = [] {
    const char* e = getenv("CQR_GEMM_NPAIR");
    return e ? atoi(e) : 1;
  }();
  return env;
}
bool pair_n_tiles(const TcGemm* t, bool split, const TcJob& job) {
  return job.pair_n && t->kind == kF16 && !split && job.n_tiles % 2 == 0;
}

// One launch of the tensor-core kernel in the variant of the handle's mode.  split: B arrives
// as raw FP32 and is split in shared memory (GEMM1 and the first block-reorthogonalisation
// product); otherwise B comes from planes.  Stages: 3 x 64 KB (two products), 2 x 96 KB (two
// products on pairs of M tiles), 6 x 32 KB (one product), 4 x 48 KB (BF16, one product, raw
// FP32 B of 64 K elements).
cudaError_t launch_mode(const TcGemm* t, bool split, const TcMaps& maps, const TcJob& job,
                        cudaStream_t st, int max_ctas = 0) {
  const int mc = max_ctas > 0 ? std::min(max_ctas, t->num_sms) : t->num_sms;
  const bool pdl = t->pdl && st == t->pdl_st;
  if (t->kind == kF16) {
    if (pair_m_tiles(t, split, job.m_tiles)) return launch_gemm<kF16, true, 2, 2, 2, 2>(maps, job, mc, st, pdl);
    if (pair_n_tiles(t, split, job)) return launch_gemm<kF16, false, 2, 2, 2, 1, 2>(maps, job, mc, st, pdl);
    return split ? launch_gemm<kF16, true, 3, 2, 2>(maps, job, mc, st, pdl)
                 : launch_gemm<kF16, false, 3, 2, 2>(maps, job, mc, st, pdl);
  }
  if (t->kind == kTF32) return launch_gemm<kTF32, false, 6, 1, 1>(maps, job, mc, st, pdl);
  if (t->nplanes == 2)
    return split ? launch_gemm<kBF16, true, 3, 2, 2>(maps, job, mc, st, pdl)
                 : launch_gemm<kBF16, false, 3, 2, 2>(maps, job, mc, st, pdl);
  return split ? launch_gemm<kBF16, true, 4, 1, 2>(maps, job, mc, st, pdl)
               : launch_gemm<kBF16, false, 6, 1, 1>(maps, job, mc, st, pdl);
}

template <typename P>
P* pl(void* p) { return static_cast<P*>(p); }

int64_t round_to(int64_t x, int64_t a) { return (x + a - 1) / a * a; }

int kind_of(int mode) {
  return mode == CQR_MMA_3XTF32 ? kF16 : mode == CQR_MMA_TF32 ? kTF32 : kBF16;
}

// FP16 scale of the orthonormal columns: |q| <= 1, with room for a factor of 16.
constexpr float kQScale = 4096.f;
float q_scale(const TcGemm* t) { return t->kind == kF16 ? kQScale : 1.f; }
float q_inv(const TcGemm* t) { return t->kind == kF16 ? 1.f / kQScale : 1.f; }
const float* inv_of(const TcGemm* t, int64_t j) { return t->kind == kF16 ? t->ci + j : nullptr; }

// f(value of the plane type)
template <typename F>
cudaError_t with_plane(const TcGemm* t, F f) {
  if (t->kind == kF16) return f(__half{});
  if (t->kind == kBF16) return f(__nv_bfloat16{});
  return f(float{});
}

}  // namespace


bool tc_available() { return true; }

size_t tc_panel_bytes(int64_t, int) { return 0; }

size_t tc_workspace_bytes(int mode, int64_t M, int64_t N, int64_t n, int b, int reorth_block) {
  const bool w16 = kind_of(mode) != kTF32;
  const size_t pe = w16 ? 2 : 4;
  const int64_t KE = w16 ? 64 : 32;
  const int64_t bkp = round_to(b, KE);
  const int64_t ldk = round_to(M, 32);
  const int64_t akc = std::max<int64_t>(bkp, round_to(b, BM));
  const int64_t ldrow = round_to(n, 64);
  size_t s = 0;
  s += 4 * al256((size_t)ldk * akc * pe);            // Ak hi/lo, two buffers
  s += 4 * al256((size_t)M * bkp * pe);              // At hi/lo, two buffers
  s += 4 * al256((size_t)bkp * N * pe);              // Rbar planes, two contexts
  s += 2 * al256((size_t)kMaxSplits * bkp * N * 4);  // split-K partials (FP32), two contexts
  if (reorth_block) {
    s += 2 * al256((size_t)M * ldrow * pe);      // row-major computed columns hi/lo
    s += 2 * al256((size_t)ldrow * akc * pe);    // S planes
  }
  if (kind_of(mode) == kF16) s += 5 * al256((size_t)N * 4);  // column scales
  return s;
}

TcGemm* tc_create(int mode, int64_t M, int64_t N, int64_t n, int64_t b, float* Q, int64_t ldq,
                  void* ws, int num_sms, int reorth_block, cudaStream_t st) {
  TcGemm* t = new (std::nothrow) TcGemm();
  if (!t) return nullptr;
  t->mode = mode;
  t->kind = kind_of(mode);
  t->nplanes = (mode == CQR_MMA_3XTF32 || mode == CQR_MMA_BF16X3) ? 2 : 1;
  t->KE = t->kind == kTF32 ? 32 : 64;
  t->pe = t->kind == kTF32 ? 4 : 2;
  t->M = M;
  t->N = N;
  t->b = b;
  t->bkp = round_to(b, t->KE);
  t->ldq = ldq;
  t->ldk = round_to(M, 32);
  t->Q = Q;
  t->num_sms = num_sms;
  const int64_t akc = std::max<int64_t>(t->bkp, round_to(b, BM));
  const size_t pe = t->pe;
  char* p = static_cast<char*>(ws);
  auto take = [&](size_t bytes) { char* r = p; p += al256(bytes); return static_cast<void*>(r); };
  for (int u = 0; u < 2; ++u) {
    t->Ak_hi[u] = take((size_t)t->ldk * akc * pe);
    t->Ak_lo[u] = take((size_t)t->ldk * akc * pe);
    t->At_hi[u] = take((size_t)M * t->bkp * pe);
    t->At_lo[u] = take((size_t)M * t->bkp * pe);
    t->Bh[u] = take((size_t)t->bkp * N * pe);
    t->Bl[u] = take((size_t)t->bkp * N * pe);
    t->P[u] = static_cast<float*>(take((size_t)kMaxSplits * t->bkp * N * 4));
  }
  t->n = n;
  t->ldrow = round_to(n, 64);
  t->Qr_hi = t->Qr_lo = t->Sh = t->Sl = nullptr;
  if (reorth_block) {
    t->Qr_hi = take((size_t)M * t->ldrow * pe);
    t->Qr_lo = take((size_t)M * t->ldrow * pe);
    t->Sh = take((size_t)t->ldrow * akc * pe);
    t->Sl = take((size_t)t->ldrow * akc * pe);
  }
  t->cs = t->ci = t->ri = nullptr;
  t->cm[0] = t->cm[1] = nullptr;
  if (t->kind == kF16) {
    t->cm[0] = static_cast<unsigned*>(take((size_t)N * 4));
    t->cm[1] = static_cast<unsigned*>(take((size_t)N * 4));
    t->ri = static_cast<float*>(take((size_t)N * 4));
    t->cs = static_cast<float*>(take((size_t)N * 4));
    t->ci = static_cast<float*>(take((size_t)N * 4));
  }
  const int kd = t->kind;
  const uint32_t KE = (uint32_t)t->KE;
  bool ok = true;
  ok &= encode_2d(&t->tm_q_b, Q, kTF32, (uint64_t)M, (uint64_t)N, (uint64_t)ldq * 4, 32, BN);
  ok &= encode_2d(&t->tm_q_c, Q, kTF32, (uint64_t)M, (uint64_t)N, (uint64_t)ldq * 4, 32, 32);
  for (int u = 0; u < 2; ++u) {
    ok &= encode_2d(&t->tm_ak[u][0], t->Ak_hi[u], kd, (uint64_t)M, (uint64_t)akc, (uint64_t)t->ldk * pe, KE, BM);
    ok &= encode_2d(&t->tm_ak[u][1], t->Ak_lo[u], kd, (uint64_t)M, (uint64_t)akc, (uint64_t)t->ldk * pe, KE, BM);
    ok &= encode_2d(&t->tm_at[u][0], t->At_hi[u], kd, (uint64_t)t->bkp, (uint64_t)M, (uint64_t)t->bkp * pe, KE, BM);
    ok &= encode_2d(&t->tm_at[u][1], t->At_lo[u], kd, (uint64_t)t->bkp, (uint64_t)M, (uint64_t)t->bkp * pe, KE, BM);
    ok &= encode_2d(&t->tm_bh[u][0], t->Bh[u], kd, (uint64_t)t->bkp, (uint64_t)N, (uint64_t)t->bkp * pe, KE, BN);
    ok &= encode_2d(&t->tm_bh[u][1], t->Bl[u], kd, (uint64_t)t->bkp, (uint64_t)N, (uint64_t)t->bkp * pe, KE, BN);
  }
  if (reorth_block) {
    ok &= encode_2d(&t->tm_qr[0], t->Qr_hi, kd, (uint64_t)t->ldrow, (uint64_t)M, (uint64_t)t->ldrow * pe, KE, BM);
    ok &= encode_2d(&t->tm_qr[1], t->Qr_lo, kd, (uint64_t)t->ldrow, (uint64_t)M, (uint64_t)t->ldrow * pe, KE, BM);
    ok &= encode_2d(&t->tm_s[0], t->Sh, kd, (uint64_t)t->ldrow, (uint64_t)akc, (uint64_t)t->ldrow * pe, KE, BN);
    ok &= encode_2d(&t->tm_s[1], t->Sl, kd, (uint64_t)t->ldrow, (uint64_t)akc, (uint64_t)t->ldrow * pe, KE, BN);
  }
  if (!ok) {
    delete t;
    return nullptr;
  }
  return t;
}

void tc_destroy(TcGemm* t) { delete t; }

void tc_set_status(TcGemm* t, int* status) { t->status = status; }

void tc_set_pdl_stream(TcGemm* t, bool on, cudaStream_t st) {
  t->pdl = on;
  t->pdl_st = st;
}

namespace {
// Split-K factor of a product with m1 x n1 output tiles and K = M rows: the count s whose
// launch finishes first on `ctas` persistent CTAs, i.e. the least (waves of work units) x
// (K blocks per unit), each unit one tile and one K chunk; a split adds partial-sum traffic,
// so each split costs 2% more and ties go to fewer splits.
// K blocks per work unit for `tiles` output tiles and `kblocks` K blocks on `ctas` CTAs, at
// most max_splits chunks (see tc_splits).
int64_t best_kchunk(int64_t tiles, int64_t kblocks, int ctas, int max_splits) {
  int64_t best_kc = kblocks;
  double best = -1.0;
  for (int s = 1; s <= max_splits && s <= kblocks; ++s) {
    const int64_t kc = (kblocks + s - 1) / s;
    const int64_t units = tiles * ((kblocks + kc - 1) / kc);
    const int64_t waves = (units + ctas - 1) / ctas;
    const double cost = (double)waves * (double)kc * (1.0 + 0.02 * s);
    if (best < 0.0 || cost < best) {
      best = cost;
      best_kc = kc;
    }
  }
  return best_kc;
}

int tc_splits(const TcGemm* t, int m1, int n1, int64_t* kchunk, int max_ctas = 0) {
  const int ctas = max_ctas > 0 ? std::min(max_ctas, t->num_sms) : t->num_sms;
  const int64_t kblocks = (t->M + t->KE - 1) / t->KE;
  // work units of the GEMM1-shaped launch (pairs of M tiles where launch_mode pairs them)
  const int units_m = pair_m_tiles(t, true, m1) ? m1 / 2 : m1;
  *kchunk = best_kchunk((int64_t)units_m * n1, kblocks, ctas, kMaxSplits) * t->KE;
  return (int)((t->M + *kchunk - 1) / *kchunk);
}
}  // namespace

// The largest magnitudes of all columns as they are before the panel of parity `buf`; each update leaves
// those of its columns for the next panel.
cudaError_t tc_begin(TcGemm* t, int buf, cudaStream_t st) {
  if (t->kind != kF16) return cudaSuccess;
  return launch_k(k_col_max, dim3((unsigned)t->N), dim3(256), 0, st, t->pdl && st == t->pdl_st,
                  (const float*)t->Q, t->ldq, t->M, t->cm[buf]);
}

namespace {
cudaError_t split_panel(TcGemm* t, int64_t kb, int bk, bool finished, const float* cscale, int buf,
                        cudaStream_t st) {
  const int bkp = (int)t->bkp;  // the planes' stride in the tensor maps, also for a narrower last panel
  const int m1 = (bk + BM - 1) / BM;
  void* qh = finished ? t->Qr_hi : nullptr;
  const int qcols = qh ? (int)(round_to(kb + bk, t->KE) - kb) : 0;  // to the end of a stage of K
  dim3 grd((unsigned)((t->M + 31) / 32), (unsigned)((std::max({bkp, m1 * BM, qcols}) + 31) / 32));
  const bool pdl = t->pdl && st == t->pdl_st;
  const float* q0 = t->Q + kb * t->ldq;
  return with_plane(t, [&](auto tag) {
    using P = decltype(tag);
    return launch_k(k_split_panel<P>, grd, dim3(256), 0, st, pdl, q0, t->ldq, t->M, bk, bkp,
                    (int)(m1 * BM), t->nplanes, pl<P>(t->Ak_hi[buf]), pl<P>(t->Ak_lo[buf]), t->ldk,
                    pl<P>(t->At_hi[buf]), pl<P>(t->At_lo[buf]), pl<P>(qh), pl<P>(t->Qr_lo), t->ldrow, kb,
                    qcols, q_scale(t), cscale);
  });
}
}  // namespace

// 1. split the finished panel Q[:, kb : kb+bk] into the operand planes of both GEMMs (and, with
//    block reorthogonalisation on, into the row-major computed columns)
cudaError_t tc_split_panel(TcGemm* t, int64_t kb, int bk, int buf, cudaStream_t st) {
  return split_panel(t, kb, bk, true, nullptr, buf, st);
}

bool tc_has_block_reorth(const TcGemm* t) { return t->Qr_hi != nullptr; }

// Row-major planes of one rectangle of Q (rows r0.., columns c0.. below the computed-column
// count) rebuilt after a recovery changed it.
cudaError_t tc_refresh_rect(TcGemm* t, int64_t r0, int64_t nr, int64_t c0, int64_t nc, cudaStream_t st) {
  if (!t->Qr_hi || nr <= 0 || nc <= 0) return cudaSuccess;
  const dim3 grd((unsigned)((nr + 31) / 32), (unsigned)((nc + 31) / 32));
  return with_plane(t, [&](auto tag) {
    using P = decltype(tag);
    k_refresh_rect<P><<<grd, 256, 0, st>>>(t->Q, t->ldq, r0, (int)nr, c0, (int)nc, t->nplanes,
                                           pl<P>(t->Qr_hi), pl<P>(t->Qr_lo), t->ldrow, q_scale(t));
    return cudaGetLastError();
  });
}

// 2. GEMM1, split-K over the M rows: partials P[s] = Qbar^T Q[:, j0 : j0+w]
namespace {
// bmax: FP16, the largest magnitudes of the columns j0.. of Q (nullptr: orthonormal columns)
cudaError_t gemm_rbar(TcGemm* t, int bk, int64_t j0, int64_t w, const unsigned* bmax, int buf, int ctx,
                      int max_ctas, cudaStream_t st) {
  const int three = t->nplanes == 2;
  const int bkp = (int)t->bkp;
  const int m1 = (bk + BM - 1) / BM;
  const int n1 = (int)((w + BN - 1) / BN);
  int64_t kchunk = 0;
  const int splits = tc_splits(t, m1, n1, &kchunk, max_ctas);
  TcMaps maps;
  maps.a[0] = t->tm_ak[buf][0];
  maps.a[1] = t->tm_ak[buf][1];
  maps.b[0] = t->tm_q_b;
  maps.b[1] = t->tm_q_b;
  TcJob job{};
  job.nprod = three ? 3 : 1;
  // TF32 reads the raw FP32 words directly with one product; every other mode splits B
  const bool split = three || t->kind != kTF32;
  job.epi = 0;
  job.m_tiles = m1;
  job.n_tiles = n1;
  job.splits = splits;
  job.a_row0 = 0;
  job.b_row0 = j0;
  job.k0 = 0;
  job.kchunk = kchunk;
  job.K = t->M;
  job.mrows = bk;
  job.ncols = w;
  job.out = t->P[ctx];
  job.ldo = bkp;
  job.split_stride = (int64_t)bkp * w;
  job.bmax = bmax;
  job.bconst = q_scale(t);
  job.status = t->status;
  return launch_mode(t, split, maps, job, st, max_ctas);
}
}  // namespace

cudaError_t tc_gemm_rbar(TcGemm* t, int bk, int64_t j0, int64_t w, int buf, int ctx, int max_ctas,
                         cudaStream_t st) {
  return gemm_rbar(t, bk, j0, w, t->kind == kF16 ? t->cm[buf] + j0 : nullptr, buf, ctx, max_ctas, st);
}

// 3. reduce the partials into R[kb.., j0..] and GEMM2's B planes
cudaError_t tc_reduce(TcGemm* t, int64_t kb, int bk, int64_t j0, int64_t w, float* R, int64_t ldr,
                      int buf, int ctx, int max_ctas, cudaStream_t st) {
  const int bkp = (int)t->bkp;
  const int m1 = (bk + BM - 1) / BM;
  const int n1 = (int)((w + BN - 1) / BN);
  int64_t kchunk = 0;
  const int splits = tc_splits(t, m1, n1, &kchunk, max_ctas);
  const int64_t total = (int64_t)bkp * w;
  const int blocks = (int)std::min<int64_t>(4096, (total + 255) / 256);
  const bool pdl = t->pdl && st == t->pdl_st;
  const float* P = t->P[ctx];
  float* Rd = R + kb + j0 * ldr;
  if (t->kind == kF16)
    return launch_k(k_tc_reduce_f16, dim3((unsigned)((w + 7) / 8)), dim3(256), 0, st, pdl, P, splits,
                    (int64_t)bkp * w, (int64_t)bkp, bk, bkp, w, Rd, ldr, pl<__half>(t->Bh[ctx]),
                    pl<__half>(t->Bl[ctx]), q_inv(t), (const unsigned*)(t->cm[buf] + j0), t->ri + j0,
                    t->cm[buf ^ 1] + j0);
  auto go = [&](auto tag) {
    using P_ = decltype(tag);
    return launch_k(k_tc_reduce<P_>, dim3(blocks), dim3(256), 0, st, pdl, P, splits, (int64_t)bkp * w,
                    (int64_t)bkp, bk, bkp, w, Rd, ldr, t->nplanes, pl<P_>(t->Bh[ctx]),
                    pl<P_>(t->Bl[ctx]));
  };
  return t->kind == kBF16 ? go(__nv_bfloat16{}) : go(float{});
}

// 4. GEMM2: Q[:, j0 : j0+w] -= Qbar Rbar (M tiles over rows, N tiles over trailing columns)
cudaError_t tc_gemm_update(TcGemm* t, int bk, int64_t j0, int64_t w, int buf, int ctx, int max_ctas,
                           cudaStream_t st) {
  const int three = t->nplanes == 2;
  const int64_t kk = round_to(bk, t->KE);  // planes are zero from bk to there
  TcMaps maps;
  maps.a[0] = t->tm_at[buf][0];
  maps.a[1] = t->tm_at[buf][1];
  maps.b[0] = t->tm_bh[ctx][0];
  maps.b[1] = t->tm_bh[ctx][1];
  TcJob job{};
  job.nprod = three ? 3 : 1;
  job.epi = 1;
  job.m_tiles = (int)((t->M + BM - 1) / BM);
  job.n_tiles = (int)((w + BN - 1) / BN);
  job.splits = 1;
  job.a_row0 = 0;
  job.b_row0 = 0;
  job.k0 = 0;
  job.kchunk = kk;
  job.K = kk;
  job.mrows = t->M;
  job.ncols = w;
  job.out = t->Q + j0 * t->ldq;
  job.ldo = t->ldq;
  job.split_stride = 0;
  job.status = t->status;
  job.c_col0 = j0;
  job.oconst = q_inv(t);
  if (t->kind == kF16) {
    job.oinv = t->ri + j0;
    job.cmax = t->cm[buf ^ 1] + j0;
    maps.c = t->tm_q_c;
    return launch_gemm<kF16, false, 2, 2, 2, 1, 1, true>(
        maps, job, max_ctas > 0 ? std::min(max_ctas, t->num_sms) : t->num_sms, st,
        t->pdl && st == t->pdl_st);
  }
  maps.c = t->tm_q_b;
  job.prefetch_c = 1;
  return launch_mode(t, false, maps, job, st, max_ctas);
}

// Block reorthogonalisation of panel kb .. kb+bk-1 against columns 0 .. kb-1 (four
// launches, five with FP16 operands: the scales of the panel's columns as they are now, split
// the panel, S^T = Qbar^T Q[:, 0:kb] split-K on the tensor cores, reduce
// into R and S, Qbar -= Qrows S on the tensor cores).
cudaError_t tc_block_reorth(TcGemm* t, int64_t kb, int bk, float* R, int64_t ldr, int buf,
                            cudaStream_t st, int* launches) {
  *launches = 0;
  if (!t->Qr_hi || kb <= 0) return cudaSuccess;
  *launches = 4;
  cudaError_t e = cudaSuccess;
  const float* ps = nullptr;
  if (t->kind == kF16) {
    ++*launches;
    e = launch_k(k_col_scale, dim3((unsigned)bk), dim3(256), 0, st, t->pdl && st == t->pdl_st,
                 (const float*)(t->Q + kb * t->ldq), t->ldq, t->M, t->cs + kb, t->ci + kb);
    if (e != cudaSuccess) return e;
    ps = t->cs + kb;
  }
  e = split_panel(t, kb, bk, false, ps, buf, st);
  if (e != cudaSuccess) return e;
  e = gemm_rbar(t, bk, 0, kb, nullptr, buf, 0, 0, st);  // partials of S^T (bk x kb), context 0
  if (e != cudaSuccess) return e;
  const int KE = t->KE;
  const int bkp = (int)t->bkp;
  const int m1 = (bk + BM - 1) / BM;
  const int n1 = (int)((kb + BN - 1) / BN);
  int64_t kchunk = 0;
  const int splits = tc_splits(t, m1, n1, &kchunk);
  const int64_t kbp = round_to(kb, KE);
  {
    const dim3 blocks((unsigned)((bk + 31) / 32), (unsigned)((kbp + 31) / 32));
    const bool pdl = t->pdl && st == t->pdl_st;
    const float* P0 = t->P[0];
    e = with_plane(t, [&](auto tag) {
      using P = decltype(tag);
      return launch_k(k_tc_reduce_t<P>, blocks, dim3(256), 0, st, pdl, P0, splits, (int64_t)bkp * kb,
                      (int64_t)bkp, bk, kb, kbp, R, ldr, t->nplanes, pl<P>(t->Sh), pl<P>(t->Sl),
                      t->ldrow, q_inv(t), inv_of(t, kb));
    });
    if (e != cudaSuccess) return e;
  }
  TcMaps maps;
  maps.a[0] = t->tm_qr[0];
  maps.a[1] = t->tm_qr[1];
  maps.b[0] = t->tm_s[0];
  maps.b[1] = t->tm_s[1];
  TcJob job{};
  job.nprod = t->nplanes == 2 ? 3 : 1;
  job.epi = 1;
  job.m_tiles = (int)((t->M + BM - 1) / BM);
  job.n_tiles = (bk + BN - 1) / BN;
  // Split K (the kb computed columns) when that makes the launch finish sooner on the SMs
  // (too few M x bk output tiles, or a last wave mostly idle); the partials go to P (capacity
  // kMaxSplits * bkp * N floats) and are subtracted in a fixed order, so the result does not
  // depend on the schedule.
  const int64_t kblk = kbp / KE;
  job.pair_n = npair_level() >= 1 ? 1 : 0;
  job.oconst = q_inv(t);
  job.oinv = inv_of(t, kb);
  const bool np2 = pair_n_tiles(t, false, job);
  const int tiles2 = job.m_tiles * (job.n_tiles / (np2 ? 2 : 1));
  const int64_t cap = std::min<int64_t>(kMaxSplits, (int64_t)kMaxSplits * t->bkp * t->N /
                                                        (t->M * (int64_t)bk));
  const int64_t kchunk2 = best_kchunk(tiles2, kblk, t->num_sms, (int)std::max<int64_t>(1, cap)) * KE;
  const int splits2 = (int)((kbp + kchunk2 - 1) / kchunk2);
  job.splits = splits2;
  job.a_row0 = 0;
  job.b_row0 = 0;
  job.k0 = 0;
  job.kchunk = kchunk2;
  job.K = kbp;
  job.mrows = t->M;
  job.ncols = bk;
  job.status = t->status;
  if (splits2 == 1) {
    job.epi = 1;
    job.out = t->Q + kb * t->ldq;
    job.ldo = t->ldq;
    job.split_stride = 0;
  } else {
    job.epi = 0;
    job.out = t->P[0];
    job.ldo = t->M;
    job.split_stride = t->M * (int64_t)bk;
  }
  e = launch_mode(t, false, maps, job, st);
  if (e != cudaSuccess || splits2 == 1) return e;
  ++*launches;
  const int64_t total = t->M * (int64_t)bk;
  const int blocks = (int)std::min<int64_t>((int64_t)t->num_sms * 8, (total + 255) / 256);
  const bool pdl = t->pdl && st == t->pdl_st;
  return launch_k(k_tc_sub_partials, dim3(blocks), dim3(256), 0, st, pdl, (const float*)t->P[0], splits2,
                  t->M, (int64_t)bk, t->Q + kb * t->ldq, t->ldq, q_inv(t), inv_of(t, kb));
}

// General C -= op(A) B in 3xTF32 on the tensor cores (the large products of the reverse mode).
// op(A) is A^T (A: K x M column-major) when a_trans, else A (M x K column-major); B is K x N
// column-major, C is M x N column-major.  A goes through the operand split into hi / lo
// planes (K-major: column-major for A^T, row-major for A); B is loaded raw and split in shared
// memory.  One CTA per 128 x 128 output tile (at most the SMs, persistent), no split over K.
// Returns cudaErrorInvalidValue (nothing launched) when a tensor-map rule is not met: B and C
// 16-byte aligned, ldb a multiple of 4.
size_t tc_gemm_sub_planes(bool a_trans, int64_t M, int64_t K) {
  return a_trans ? 2 * (size_t)round_to(K, 32) * (size_t)M : 2 * (size_t)M * (size_t)round_to(K, 32);
}

cudaError_t tc_gemm_sub3(bool a_trans, const float* A, int64_t lda, const float* B, int64_t ldb,
                         float* C, int64_t ldc, int64_t M, int64_t N, int64_t K, float* planes,
                         int num_sms, int* status, cudaStream_t st) {
  if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
  if ((reinterpret_cast<uintptr_t>(B) & 15) || (ldb % 4) || (reinterpret_cast<uintptr_t>(planes) & 15))
    return cudaErrorInvalidValue;
  const int64_t kp = round_to(K, 32);
  float* hi = planes;
  TcMaps maps;
  bool ok = true;
  if (a_trans) {
    // planes of A (K x M): column-major, ld kp; rows of op(A) are columns of A
    float* lo = hi + kp * M;
    const dim3 grd((unsigned)((K + 31) / 32), (unsigned)((M + 31) / 32));
    k_split_panel<float><<<grd, 256, 0, st>>>(A, lda, K, (int)M, 0, (int)M, 2, hi, lo, kp, nullptr,
                                              nullptr, nullptr, nullptr, 0, 0, 0, 1.f, nullptr);
    ok &= encode_2d(&maps.a[0], hi, kTF32, (uint64_t)K, (uint64_t)M, (uint64_t)kp * 4, 32, BM);
    ok &= encode_2d(&maps.a[1], lo, kTF32, (uint64_t)K, (uint64_t)M, (uint64_t)kp * 4, 32, BM);
  } else {
    // planes of A (M x K): row-major, row stride kp
    float* lo = hi + M * kp;
    const dim3 grd((unsigned)((M + 31) / 32), (unsigned)((kp + 31) / 32));
    k_split_panel<float><<<grd, 256, 0, st>>>(A, lda, M, (int)K, (int)kp, 0, 2, nullptr, nullptr, 0, hi,
                                              lo, nullptr, nullptr, 0, 0, 0, 1.f, nullptr);
    ok &= encode_2d(&maps.a[0], hi, kTF32, (uint64_t)kp, (uint64_t)M, (uint64_t)kp * 4, 32, BM);
    ok &= encode_2d(&maps.a[1], lo, kTF32, (uint64_t)kp, (uint64_t)M, (uint64_t)kp * 4, 32, BM);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  ok &= encode_2d(&maps.b[0], const_cast<float*>(B), kTF32, (uint64_t)K, (uint64_t)N, (uint64_t)ldb * 4, 32, BN);
  maps.b[1] = maps.b[0];
  if (!ok) return cudaErrorInvalidValue;
  TcJob job{};
  job.nprod = 3;
  job.epi = 1;
  job.m_tiles = (int)((M + BM - 1) / BM);
  job.n_tiles = (int)((N + BN - 1) / BN);
  job.splits = 1;
  job.a_row0 = 0;
  job.b_row0 = 0;
  job.k0 = 0;
  job.kchunk = kp;
  job.K = K;
  job.mrows = M;
  job.ncols = N;
  job.out = C;
  job.ldo = ldc;
  job.split_stride = 0;
  job.status = status;
  return launch_gemm<kTF32, true, 3, 2, 2>(maps, job, num_sms, st, false);
}

cudaError_t bounds_take_tc(int* code, int* site) { return bounds_take_here(code, site); }

}  // namespace cqr
