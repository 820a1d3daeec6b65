// Row-wise Top-K of a [rows][cols] fp32 matrix (largest value first, lowest column on ties), used for the retrieval
// scores (one row) and for the per-position Top-K of the verify logits that feeds the successor table of the
// Token-Recycling-style drafter.
#include "kernels.h"

namespace ts {

// Selection in two levels, both with the same rule (largest score, lowest index on ties).  First a CTA per slice of 4096
// scores: every thread sorts its 16 in registers, every warp takes the K best of its 512 from the heads of its lanes' lists
// in K rounds of two warp reductions (no barrier), and one warp merges the eight warps' lists the same way.  Then a CTA per
// row merges the slices' lists.  (14 us cold for the two kernels, K = 10 of 100 000 scores; with a block-wide reduction over all scores per round 18,
// with warp-wide rounds over unsorted registers 48.)
// cand: [rows][slices][K] (column as int bits, value) pairs, best first; out: [rows][K] pairs.
static constexpr int kSlice = 4096;
static constexpr int kSelThreads = 256;
static constexpr int kSelWarps = kSelThreads / 32;
static constexpr int kPer = kSlice / kSelThreads;   // entries per thread

// An entry as one word that orders like (score, then lower index): order-preserving map of the score above the index's
// complement; 0 = no entry (also for NaN and -inf, which are never taken).  Both zeros are the same score: -0 + 0 = +0.
typedef unsigned long long Entry;
__device__ __forceinline__ Entry entry_of(float v, int idx) {
  if (!(v > -INFINITY)) return 0ull;
  uint32_t u = __float_as_uint(v + 0.f);
  u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
  return ((Entry)u << 32) | (uint32_t)~idx;
}
__device__ __forceinline__ float2 pair_of(Entry e) {   // (column as int bits, value)
  if (e == 0ull) return make_float2(__int_as_float(0x7FFFFFFF), -INFINITY);
  const uint32_t k = (uint32_t)(e >> 32);
  return make_float2(__int_as_float((int)~(uint32_t)e), __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k));
}
// the largest entry over the warp's lanes; `mine` = whether it is this lane's
__device__ __forceinline__ Entry warp_max(Entry e, bool &mine) {
  const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(e >> 32));
  const uint32_t lo = __reduce_max_sync(0xffffffffu, (uint32_t)(e >> 32) == hi ? (uint32_t)e : 0u);
  const Entry top = ((Entry)hi << 32) | lo;
  mine = top != 0ull && e == top;   // (entries are unique)
  return top;
}
// The K best of the warp's lists, one sorted list per lane (`next()` gives its entries one by one, 0 at the end).
template <typename F>
__device__ __forceinline__ void warp_merge(F next, int K, Entry *out) {
  Entry head = next(), second = next();   // (the entry after the head is on its way when the head goes)
  for (int j = 0; j < K; ++j) {
    bool mine;
    const Entry top = warp_max(head, mine);
    if ((threadIdx.x & 31) == 0) out[j] = top;
    if (mine) {
      head = second;
      second = next();
    }
  }
}

__global__ void __launch_bounds__(kSelThreads)
topk_slice_kernel(const float *x, int N, int K, float2 *cand) {
  __shared__ Entry lists[kSelWarps][kTopMax], best[kTopMax];
  const float *scores = x + (size_t)blockIdx.y * N;          // this CTA's row
  cand += ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * K;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int base = blockIdx.x * kSlice + threadIdx.x;
  pdl_launch_dependents();
  pdl_wait();
  float v[kPer];
#pragma unroll
  for (int e = 0; e < kPer; ++e) v[e] = base + e * kSelThreads < N ? scores[base + e * kSelThreads] : -INFINITY;
  Entry a[kPer];
#pragma unroll
  for (int e = 0; e < kPer; ++e) a[e] = entry_of(v[e], base + e * kSelThreads);
  // bitonic sorting network, largest first
#pragma unroll
  for (int k = 2; k <= kPer; k <<= 1)
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1)
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        const int l = i ^ j;
        if (l > i) {
          const bool up = (i & k) == 0;   // this pair in descending order
          const Entry p = a[i], q = a[l];
          const bool swap = up ? p < q : p > q;
          a[i] = swap ? q : p;
          a[l] = swap ? p : q;
        }
      }
  // the K best of the warp: the lanes' lists by their heads
  for (int j = 0; j < K; ++j) {
    bool mine;
    const Entry top = warp_max(a[0], mine);
    if (lane == 0) lists[warp][j] = top;
    if (mine) {
#pragma unroll
      for (int e = 0; e + 1 < kPer; ++e) a[e] = a[e + 1];
      a[kPer - 1] = 0ull;
    }
  }
  __syncthreads();
  if (warp == 0) {
    int at = 0;
    warp_merge([&]() { return lane < kSelWarps && at < K ? lists[lane][at++] : 0ull; }, K, best);
    __syncwarp();
    for (int j = lane; j < K; j += 32) cand[j] = pair_of(best[j]);
  }
}

__global__ void __launch_bounds__(kSelThreads)
topk_final_kernel(const float2 *cand, int n_lists, int K, float *out, PairsOut po, const int *err) {
  __shared__ Entry lists[kSelWarps + 1][kTopMax], best[kTopMax];
  cand += (size_t)blockIdx.x * n_lists * K;
  out += (size_t)blockIdx.x * 2 * K;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int j = threadIdx.x; j < K; j += blockDim.x) lists[kSelWarps][j] = 0ull;   // (the K best so far)
  pdl_wait();
  // a thread per slice's list: every warp merges its 32, one warp the warps' lists and what earlier rounds left
  for (int l0 = 0; l0 < n_lists; l0 += kSelThreads) {
    const int l = l0 + warp * 32 + lane;
    int at = l < n_lists ? 0 : K;
    const float2 *mine = cand + (size_t)l * K;
    warp_merge([&]() { if (at >= K) return (Entry)0; const float2 c = mine[at++]; return entry_of(c.y, __float_as_int(c.x)); }, K, lists[warp]);
    __syncthreads();
    if (warp == 0) {
      int i = 0;
      warp_merge([&]() { return lane <= kSelWarps && i < K ? lists[lane][i++] : 0ull; }, K, best);
      __syncwarp();
      for (int j = lane; j < K; j += 32) lists[kSelWarps][j] = best[j];
    }
    __syncthreads();
  }
  if (threadIdx.x < K) {
    const float2 r = pair_of(lists[kSelWarps][threadIdx.x]);
    out[2 * threadIdx.x] = r.x;
    out[2 * threadIdx.x + 1] = r.y;
    if (po.host) { po.host[2 * threadIdx.x] = r.x; po.host[2 * threadIdx.x + 1] = r.y; }
  }
  if (!po.host) return;
  int32_t *tail = reinterpret_cast<int32_t *>(po.host) + 2 * kTopMax;
  if (threadIdx.x == 0) tail[0] = *err;
  __syncthreads();
  if (threadIdx.x == 0) raise_flag(tail + 1, po.number);
}

cudaError_t launch_topk_rows(const float *x, int n_rows, int n_cols, int K, float2 *cand, float *out, PairsOut po,
                             const int *err, cudaStream_t st) {
  if (K < 1 || K > kTopMax || n_rows < 1 || n_cols < 1) return cudaErrorInvalidValue;
  const int slices = (n_cols + kSlice - 1) / kSlice;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(slices, n_rows);
  cfg.blockDim = dim3(kSelThreads);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, topk_slice_kernel, x, n_cols, K, cand);
  if (e != cudaSuccess) return e;
  cfg.gridDim = dim3(n_rows);
  return cudaLaunchKernelEx(&cfg, topk_final_kernel, (const float2 *)cand, slices, K, out, po, err);
}

}  // namespace ts
