// Top-K retrieval over the datastore's hidden states (Section 4.3, Eq. 3): sim = cosine similarity between the
// query's hidden state and each historical invocation's, the K most similar entries become the candidates of
// the suffix match.
//
// cosine_scores_kernel: one pass over N x d x 2 bytes, bound by HBM.  One CTA per SM; every warp walks the store in pieces of
// a few neighbouring entries (about 16 KB), each fetched by one bulk copy into a buffer of its own: long contiguous
// requests and no register per byte in flight; while a warp works on its piece the other seven's are on their way.  The
// 100 000 x 4096 store in 127 us (6.45 TB/s, the copy rate); a warp per entry with 16-byte loads took 150, four entries per
// warp 145; rings of 2 and 3 buffers for six and four warps are slower (5 - 9 %: the arithmetic of fewer warps), twelve
// warps too.  Entries are worked on in pairs, so that a piece of the query is read from shared memory once for two.  fp32
// dot product and squared norm.
// The K best scores are then taken by the row Top-K kernels (topk.cu).
#include <algorithm>

#include "kernels.h"

namespace ts {

static constexpr int kCosWarps = 8;
static constexpr int kCosPieceBytes = 16384;

__device__ __forceinline__ void cos_add(const uint4 &raw, const float4 &q0, const float4 &q1, float2 &dot, float2 &hh) {
  const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
  const float2 q[4] = {make_float2(q0.x, q0.y), make_float2(q0.z, q0.w), make_float2(q1.x, q1.y), make_float2(q1.z, q1.w)};
#pragma unroll
  for (int i = 0; i < 4; ++i) {   // (a bf16 is the upper half of an fp32)
    const float2 a = make_float2(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xFFFF0000u));
    dot = fma2(a, q[i], dot);
    hh = fma2(a, a, hh);
  }
}

// q_dev != nullptr: the query as fp32 [d]; else the bf16 (hi[, lo]) planes of a row of the last step's hidden state.
// piece = entries per stage; shared memory: the query (elements 8c .. 8c + 3 of all c, then 8c + 4 .. 8c + 7: reads
// without bank conflicts), then a piece each for the first `bufs` warps (wide entries leave room for fewer than eight; all
// warps bring the query in: with two warps doing it a store of one entry of 16384 took 15 us longer).
__global__ void __launch_bounds__(32 * kCosWarps)
cosine_scores_kernel(const __nv_bfloat16 *H, int N, int d, int piece, int bufs, const float *q_dev, const __nv_bfloat16 *q_planes,
                     int plane_stride, int planes, float *scores, int *err) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ float red[kCosWarps];
  __shared__ uint64_t bars[kCosWarps];
  pdl_launch_dependents();   // (the Top-K kernel waits for this one's end)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n_chunks = d / 8;                       // 8 bf16 = 16 bytes
  float4 *qa = reinterpret_cast<float4 *>(smem), *qb = qa + n_chunks;
  const uint32_t row_bytes = 2u * d, piece_bytes = piece * row_bytes;
  const uint8_t *src = smem + (size_t)d * 4 + (size_t)warp * piece_bytes;
  const uint32_t bar = smem_u32(&bars[warp]);
  const int n_pieces = (N + piece - 1) / piece, step = gridDim.x * bufs, p0 = warp < bufs ? blockIdx.x * bufs + warp : n_pieces;
  const uint64_t pol = policy_evict_first();
  auto fetch = [&](int p) {   // (one lane)
    const uint32_t bytes = min(piece, N - p * piece) * row_bytes;
    mbar_expect_tx(bar, bytes);
    bulk_load(smem_u32(src), H + (size_t)p * piece * d, bytes, bar, pol);
  };
  if (lane == 0) {
    mbar_init(bar, 1);
    fence_barrier_init();
    if (p0 < n_pieces) fetch(p0);
  }
  float qq = 0.f;
  for (int i = threadIdx.x; i < d; i += blockDim.x) {
    float v;
    if (q_dev) v = q_dev[i];
    else v = __bfloat162float(q_planes[i]) + (planes == 2 ? __bfloat162float(q_planes[plane_stride + i]) : 0.f);
    reinterpret_cast<float *>((i & 4) ? qb : qa)[(i >> 3) * 4 + (i & 3)] = v;
    qq += v * v;
  }
  qq = warp_sum(qq);
  if (lane == 0) red[warp] = qq;
  __syncthreads();
  qq = 0.f;
  for (int w = 0; w < kCosWarps; ++w) qq += red[w];
  uint32_t ph = 0;
  for (int p = p0; p < n_pieces; p += step, ph ^= 1u) {
    if (!__all_sync(0xffffffffu, mbar_wait(bar, ph))) {
      if (lane == 0) atomicExch(err, DEV_TIMEOUT_FULL);
      break;
    }
    const int e0 = p * piece, rows = min(piece, N - e0);
    for (int r = 0; r < rows; r += 2) {
      // (the odd last entry of a piece is its pair's second too; nothing is kept of that)
      const uint4 *r0 = reinterpret_cast<const uint4 *>(src + (size_t)r * row_bytes);
      const uint4 *r1 = r + 1 < rows ? r0 + n_chunks : r0;
      float2 d0 = make_float2(0.f, 0.f), d1 = d0, n0 = d0, n1 = d0;
#pragma unroll 4
      for (int c = lane; c < n_chunks; c += 32) {
        const float4 a = qa[c], b = qb[c];
        cos_add(r0[c], a, b, d0, n0);
        cos_add(r1[c], a, b, d1, n1);
      }
      const float dot0 = d0.x + d0.y, dot1 = d1.x + d1.y, h0 = n0.x + n0.y, h1 = n1.x + n1.y;
      // four sums over the warp in six shuffles: half the lanes go on with either entry, then with dot product or norm
      const bool second = lane & 16, norm = lane & 8;
      float dd = (second ? dot1 : dot0) + __shfl_xor_sync(0xffffffffu, second ? dot0 : dot1, 16);
      float nn = (second ? h1 : h0) + __shfl_xor_sync(0xffffffffu, second ? h0 : h1, 16);
      float v = (norm ? nn : dd) + __shfl_xor_sync(0xffffffffu, norm ? dd : nn, 8);
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      dd = v;
      nn = __shfl_xor_sync(0xffffffffu, v, 8);
      if ((lane & 15) == 0 && r + (lane >> 4) < rows)
        scores[e0 + r + (lane >> 4)] = (nn > 0.f && qq > 0.f) ? dd * rsqrtf(nn) * rsqrtf(qq) : -2.f;   // a zero vector ranks last
    }
    __syncwarp();   // (all lanes have read the piece)
    if (lane == 0 && p + step < n_pieces) fetch(p + step);
  }
}

cudaError_t launch_topk_cosine(const __nv_bfloat16 *H, int N, int d, const float *q_dev, const __nv_bfloat16 *q_planes,
                               int plane_stride, int planes, int K, float *scores, int n_sms, PairsOut po, int *err,
                               cudaStream_t st) {
  static PerDeviceOnce once;
  int dev_ = -1;
  constexpr size_t kSmem = 225 * 1024;
  if (once.needed(&dev_)) {
    cudaError_t e = cudaFuncSetAttribute(cosine_scores_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
    if (e != cudaSuccess) return e;
    once.done(dev_);
  }
  // entries per piece: about 16 KB, an even number (a single entry where a pair does not fit beside the query)
  int piece = std::max(2, kCosPieceBytes / (2 * d) / 2 * 2);
  while (piece > 1 && (size_t)d * 4 + (size_t)piece * 2 * d > kSmem) piece /= 2;
  const size_t piece_bytes = (size_t)piece * 2 * d;
  if ((size_t)d * 4 + piece_bytes > kSmem) return cudaErrorInvalidValue;
  const int bufs = (int)std::min<size_t>(kCosWarps, (kSmem - (size_t)d * 4) / piece_bytes);
  const int n_pieces = (N + piece - 1) / piece;
  cosine_scores_kernel<<<std::min((n_pieces + bufs - 1) / bufs, n_sms), 32 * kCosWarps, (size_t)d * 4 + bufs * piece_bytes, st>>>(
      H, N, d, piece, bufs, q_dev, q_planes, plane_stride, planes, scores, err);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // candidates live behind the K result pairs: scores[N + 2K ...], 2 floats per candidate
  float2 *cand = reinterpret_cast<float2 *>(scores + N + 2 * K + ((N + 2 * K) & 1));
  return launch_topk_rows(scores, 1, N, K, cand, scores + N, po, err, st);
}

}  // namespace ts
