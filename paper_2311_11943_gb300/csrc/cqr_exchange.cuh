// cqr_exchange.cuh -- sums over the CTAs of a cooperative launch through global memory (L2),
// shared by the sub-block panel (cqr_panel_blk.cu) and the least-squares solve (cqr_lstsq.cu).
//
// Sum of E values over G CTAs, the same bits in every CTA and in every run: each CTA writes its
// values to its row of a global buffer, CTA c adds the G values of entries [c E / G, (c+1) E / G)
// in a fixed order and writes the sums, every CTA reads all E sums.  Values travel as 64-bit
// words {32 bits of value, tag} (a double as two words), written and read whole, so a reader
// that finds the step's tag has the value: no flag, fence or barrier.  Tags are the running
// count of a word in global memory that the launch reads when it starts and advances when it
// ends, so no launch, and no replay of a captured launch, meets a tag of an earlier one.  One
// buffer is enough: a CTA writes its values of step k+1 only after it has all sums of step k, for
// which every value of step k was read; and a sum of step k+1 is written only after every CTA
// has sent its values of step k+1, hence has read the sums of step k.
#pragma once
#include "cqr_device.cuh"

namespace cqr {

typedef unsigned long long u64;

__device__ __forceinline__ u64 ld_rlx(const u64* p) {
  u64 v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_rlx(u64* p, u64 v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ void st_release_u32(unsigned* p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// One value as words {32 bits of value, tag}: a float is one word, a double two.
template <typename T>
struct Wire;
template <>
struct Wire<float> {
  static constexpr int kWords = 1;
  __device__ static void put(u64* p, float x, unsigned tag) {
    st_rlx(p, ((u64)tag << 32) | __float_as_uint(x));
  }
  __device__ static float value(const u64* w) { return __uint_as_float((unsigned)w[0]); }
};
template <>
struct Wire<double> {
  static constexpr int kWords = 2;
  __device__ static void put(u64* p, double x, unsigned tag) {
    const u64 b = (u64)__double_as_longlong(x);
    st_rlx(p, ((u64)tag << 32) | (unsigned)b);
    st_rlx(p + 1, ((u64)tag << 32) | (unsigned)(b >> 32));
  }
  __device__ static double value(const u64* w) {
    return __longlong_as_double((long long)((w[1] << 32) | (unsigned)w[0]));
  }
};

// Poll N words until each carries the tag (bounded): x holds a first reading, want[i] whether
// word i is wanted.  The words that are not there yet are read again together, so a thread waits
// for the last of them and not for each in turn (panels of 8192 x 8192: 7.8 -> 7.3 ms; of
// 16384 x 2048: 2.00 -> 1.88 ms, its least-squares solve 0.98 -> 0.89 ms).
template <int N>
__device__ __forceinline__ bool poll_all(const u64* const (&p)[N], u64 (&x)[N], const bool (&want)[N],
                                         unsigned tag, int* status, int site, long long limit) {
  bool missing = false;
#pragma unroll
  for (int i = 0; i < N; ++i) missing = missing || (want[i] && (unsigned)(x[i] >> 32) != tag);
  if (!missing) return true;
  const long long t0 = clock64();
  unsigned spins = 0u;
  for (;;) {
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (want[i] && (unsigned)(x[i] >> 32) != tag) x[i] = ld_rlx(p[i]);
    missing = false;
#pragma unroll
    for (int i = 0; i < N; ++i) missing = missing || (want[i] && (unsigned)(x[i] >> 32) != tag);
    if (!missing) return true;
    const long long el = clock64() - t0;
    if (el > limit) {
      set_status(status, CQR_ETIMEOUT, site);
      return false;
    }
    if (el > kPollAfterCycles && (++spins & 63u) == 0u && ld_relaxed_i32(status + ST_CODE) != 0)
      return false;
  }
}

// Buffers and step of the sums of one launch.
struct Xch {
  unsigned long long* part;  // [G][ecap] words
  unsigned long long* fin;   // [ecap] words
  int ecap;                  // words per row
  unsigned tag;
  int* status;
  long long limit;           // bound of a wait, SM cycles
};

// Start of a launch that uses `tags` steps at most: the first tag into c.tag.  False (the same in
// every thread) when an error was recorded before this CTA began (an earlier launch's, or an
// exchange of this launch that was given up): the caller leaves without sending a word.  CTA 0
// advances the count only after such an error is recorded, so a CTA that reads the advanced
// count also reads the error, and no word of an abandoned launch carries a tag of the next one.
__device__ __forceinline__ bool exchange_begin(Xch& c, unsigned* epoch, unsigned tags) {
  __shared__ unsigned sTag;
  __shared__ int sErr;
  if (threadIdx.x == 0) {  // one thread reads both, the count first
    sTag = ld_acquire_u32(epoch);
    sErr = ld_relaxed_i32(c.status + ST_CODE);
  }
  __syncthreads();
  const unsigned tag0 = sTag;
  const bool ok = sErr == 0;
  c.tag = tag0 + 1;
  if (!ok && blockIdx.x == 0 && threadIdx.x == 0) st_release_u32(epoch, tag0 + tags);
  return ok;
}

// End of the launch, from the count `first` = c.tag after exchange_begin: every CTA has read the
// count (CTA 0 has had sums that each of them sent after reading it, or the launch is being
// abandoned).
__device__ __forceinline__ void exchange_end(unsigned* epoch, unsigned first, unsigned tags) {
  if (blockIdx.x == 0 && threadIdx.x == 0) st_release_u32(epoch, first - 1u + tags);
}

// W[0, E) <- the sums over the CTAs of their W[0, E) (shared memory, as is red[NT]).  False (the
// same in every thread) when a wait ran out.  Every thread of the CTA (NT of them) calls it.
template <typename T, int NT>
__device__ __forceinline__ bool exchange(Xch& c, T* W, int E, T* red) {
  constexpr int KW = Wire<T>::kWords;
  const int G = gridDim.x, g = blockIdx.x, tid = threadIdx.x;
  __syncthreads();
  if (G == 1) return true;
  {
    u64* mine = c.part + (size_t)g * c.ecap;
    for (int e = tid; e < E; e += NT) Wire<T>::put(mine + e * KW, W[e], c.tag);
  }
  bool ok = true;
  const int chunk = (E + G - 1) / G;
  const int e0 = g * chunk, ne = max(0, min(chunk, E - e0));
  if (ne > 0) {
    // threads: entry fastest, then groups of partial rows
    int nep = 1;
    while (nep < chunk && nep < NT) nep *= 2;
    const int ng = NT / nep, grp = tid / nep;
    for (int b0 = 0; b0 < ne; b0 += nep) {
      const int e = b0 + tid % nep;
      T acc = T(0);
      if (e < ne) {
        const u64* col = c.part + (size_t)(e0 + e) * KW;
        constexpr int F = 8 / KW;  // partials in flight
        for (int r0 = grp; r0 < G && ok; r0 += F * ng) {
          u64 x[F * KW];
          const u64* p[F * KW];
          bool want[F * KW];
#pragma unroll
          for (int u = 0; u < F; ++u)
#pragma unroll
            for (int k = 0; k < KW; ++k) {
              const int i = u * KW + k;
              want[i] = r0 + u * ng < G;
              p[i] = col + (size_t)(want[i] ? r0 + u * ng : r0) * c.ecap + k;
              x[i] = want[i] ? ld_rlx(p[i]) : 0ull;
            }
          ok = poll_all<F * KW>(p, x, want, c.tag, c.status, 60, c.limit);
#pragma unroll
          for (int u = 0; u < F; ++u)
            if (want[u * KW]) acc += Wire<T>::value(x + u * KW);
        }
      }
      // the groups: within a warp by a butterfly, over the warps through shared memory
      for (int o = nep; o < 32; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (ng > 1) {
        const int step = nep < 32 ? 32 : nep;  // threads that hold one copy of the entries
        red[tid] = acc;
        __syncthreads();
        if (tid < step) {
          // lanes that repeat an entry share its rows
          const int rep = step / nep, q0 = tid / nep, ent = tid - q0 * nep;
          acc = T(0);
#pragma unroll 4
          for (int q = q0; q < NT / step; q += rep) acc += red[q * step + ent];
          for (int o = nep; o < 32; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        }
        __syncthreads();
      }
      if (grp == 0 && e < ne) Wire<T>::put(c.fin + (size_t)(e0 + e) * KW, acc, c.tag);
    }
  }
  constexpr int F = 8 / KW;  // sums in flight
  for (int b0 = 0; b0 < E; b0 += F * NT) {
    u64 x[F * KW];
    const u64* p[F * KW];
    bool want[F * KW];
#pragma unroll
    for (int u = 0; u < F; ++u)
#pragma unroll
      for (int k = 0; k < KW; ++k) {
        const int e = b0 + u * NT + tid, i = u * KW + k;
        want[i] = e < E && ok;
        p[i] = c.fin + (size_t)(want[i] ? e : 0) * KW + k;
        x[i] = want[i] ? ld_rlx(p[i]) : 0ull;
      }
    ok = ok && poll_all<F * KW>(p, x, want, c.tag, c.status, 61, c.limit);
#pragma unroll
    for (int u = 0; u < F; ++u)
      if (want[u * KW]) W[b0 + u * NT + tid] = Wire<T>::value(x + u * KW);
  }
  ++c.tag;
  return __syncthreads_and(ok) != 0;
}

}  // namespace cqr
