// Row-wise Top-K of a [rows][cols] fp32 matrix (largest value first, lowest column on ties), used for the retrieval
// scores (one row) and for the per-position Top-K of the verify logits that feeds the successor table of the
// Token-Recycling-style drafter.
#include "kernels.h"

namespace ts {

// Selection in two levels, both with the same rule (largest score, lowest index on ties).  First a CTA per slice of 4096
// scores.  Up to kBoundK: the K-th largest of a warp's 32 lane maxima is a bound that at least K of its scores reach; the
// largest bound of the CTA's warps leaves a few dozen of the slice, which are put in order by counting, for each, those above
// it.  For larger K every thread sorts its 16 in registers, every warp takes the K best of its 512 from the heads of its lanes'
// lists in K rounds of two warp reductions (no barrier), and one warp merges the eight warps' lists the same way.  Then a CTA
// per row merges the slices' lists.
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

static constexpr int kBoundK = 16;      // most K of the bounded selection
__global__ void __launch_bounds__(kSelThreads, 6)
topk_bound_kernel(const float *x, int N, int K, float2 *cand) {
  __shared__ Entry list[kSelThreads], best[kBoundK], of_warp[kSelWarps];
  __shared__ uint32_t bound, count;
  const float *scores = x + (size_t)blockIdx.y * N;          // this CTA's row
  cand += ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * K;
  const int lane = threadIdx.x & 31, base = blockIdx.x * kSlice + threadIdx.x;
  if (threadIdx.x == 0) { bound = 1u; count = 0u; }
  if (threadIdx.x < K) best[threadIdx.x] = 0ull;
  pdl_launch_dependents();
  pdl_wait();
  uint32_t u[kPer], top = 0u;   // the scores as words of the same order, 0 = none
  {
    float v[kPer];
#pragma unroll
    for (int e = 0; e < kPer; ++e) v[e] = base + e * kSelThreads < N ? scores[base + e * kSelThreads] : -INFINITY;
#pragma unroll
    for (int e = 0; e < kPer; ++e) {
      u[e] = (uint32_t)(entry_of(v[e], 0) >> 32);
      top = max(top, u[e]);
    }
  }
  auto entry = [&](int e) { return u[e] ? ((Entry)u[e] << 32) | (uint32_t)~(base + e * kSelThreads) : 0ull; };
  uint32_t mine = top, b = 0u;
  for (int j = 0; j < K; ++j) {
    b = __reduce_max_sync(0xffffffffu, mine);
    if (lane == __ffs(__ballot_sync(0xffffffffu, mine == b)) - 1) mine = 0u;
  }
  __syncthreads();
  if (lane == 0) atomicMax(&bound, b);   // (0 where the warp has fewer than K)
  __syncthreads();
  const uint32_t least = bound;
  if (__any_sync(0xffffffffu, top >= least)) {
#pragma unroll
    for (int e = 0; e < kPer; ++e) {
      const uint32_t hit = __ballot_sync(0xffffffffu, u[e] >= least);
      if (hit == 0u) continue;
      uint32_t at = 0u;
      if (lane == 0) at = atomicAdd(&count, (uint32_t)__popc(hit));
      at = __shfl_sync(0xffffffffu, at, 0) + __popc(hit & ((1u << lane) - 1u));
      if (u[e] >= least && at < kSelThreads) list[at] = entry(e);
    }
  }
  __syncthreads();
  const int n = (int)count;
  if (n <= kSelThreads) {
    if ((int)threadIdx.x < n) {
      const Entry e = list[threadIdx.x];
      int above = 0;
#pragma unroll 8
      for (int i = 0; i < n; ++i) above += list[i] > e;
      if (above < K) best[above] = e;   // (entries are unique)
    }
  } else {
    // (hundreds of equal scores: one after the other, each the largest below the one before)
    Entry last = ~0ull;
    for (int j = 0; j < K; ++j) {
      Entry e = 0ull;
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        const Entry t = entry(i);
        if (t < last && t > e) e = t;
      }
      bool is_mine;
      e = warp_max(e, is_mine);
      if (lane == 0) of_warp[threadIdx.x >> 5] = e;
      __syncthreads();
      e = 0ull;
      for (int w = 0; w < kSelWarps; ++w) e = max(e, of_warp[w]);
      if (threadIdx.x == 0) best[j] = e;
      last = e;
      __syncthreads();
    }
  }
  __syncthreads();
  if (threadIdx.x < K) cand[threadIdx.x] = pair_of(best[threadIdx.x]);
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
  pdl_launch_dependents();
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
    if (po.host) {
      float *host = po.host + (size_t)blockIdx.x * 2 * K;
      host[2 * threadIdx.x] = r.x;
      host[2 * threadIdx.x + 1] = r.y;
      if (!po.ends) __threadfence_system();   // (else raise_flag's)
    }
  }
  if (!po.host || !po.ends) return;
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
  cudaError_t e = cudaLaunchKernelEx(&cfg, K <= kBoundK ? topk_bound_kernel : topk_slice_kernel, x, n_cols, K, cand);
  if (e != cudaSuccess) return e;
  cfg.gridDim = dim3(n_rows);
  return cudaLaunchKernelEx(&cfg, topk_final_kernel, (const float2 *)cand, slices, K, out, po, err);
}

}  // namespace ts
