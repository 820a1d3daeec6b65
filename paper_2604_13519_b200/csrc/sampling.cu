// Speculative-sampling acceptance at temperature T > 0 (Appendix B.2 names speculative sampling as the acceptance
// strategy).  The drafts come from retrieval or the schema, so the draft distribution is a point mass on the drafted
// token x and the rule reads: accept x with probability p(x), p = softmax(logits / T) of the row that predicts it;
// on the first rejection emit one sample of p with x removed (renormalised) and stop; if every draft is accepted
// emit one sample of the last row's p.  Over a draft tree the children of a node are tried in node order against
// the residual of the refused ones.  The uniforms are inputs: uni[node c] decides node c, the root's draws the sample
// (the host renames a chain's uniforms accordingly).  A sample is the smallest index whose running sum of weights, in index order, exceeds
// u times the total.
#include "kernels.h"

namespace ts {

static constexpr int kStatThreads = 256;
static constexpr int kStatSlices = kSampleSlices;   // slices a row's statistics are kept in, a warp's lane each in the draw
static constexpr int kSampleThreads = 512;

// ids per slice: a multiple of 128, like V
__device__ __forceinline__ int slice_len(int V) { return (V / 128 + kStatSlices - 1) / kStatSlices * 128; }

// the row maximum, from the packed (ordered value bits, ~id) word the LM-head epilogue reduced
__device__ __forceinline__ float row_max_of(unsigned long long word) {
  const uint32_t u = (uint32_t)(word >> 32);
  return __uint_as_float((u & 0x80000000u) ? (u & 0x7FFFFFFFu) : ~u);
}

__device__ __forceinline__ float4 weights4(const float *row, int i, float mx, float inv_t) {
  const float4 v = __ldcg(reinterpret_cast<const float4 *>(row + i));
  return make_float4(__expf((v.x - mx) * inv_t), __expf((v.y - mx) * inv_t), __expf((v.z - mx) * inv_t), __expf((v.w - mx) * inv_t));
}

// sum of v over a CTA of at most 32 warps, in every thread
__device__ __forceinline__ float cta_sum(float v, float *red) {
  v = warp_sum(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  return warp_sum(lane < (int)(blockDim.x >> 5) ? red[lane] : 0.f);
}

// grid = (rows, slices / PER): sums of exp((l - max) / T) over the slices of a row, PER of them per CTA with 256 / PER threads
// each.  Short slices take a warp each (PER = 8): with a CTA per slice 400 rows of 4096 ids were 12 800 CTAs of one working
// warp, and sampling cost 16.3 us more than greedy acceptance; now 5.6 (16 384 ids: 16.6 and 6.6).
static constexpr int kWarpSlice = 512;   // ids up to which a warp takes a slice: four loads per lane
template <int PER>
__global__ void __launch_bounds__(kStatThreads)
row_expsum_kernel(const float *logits, const unsigned long long *amax, int V, float inv_t, float *part) {
  __shared__ float red[kStatThreads / 32];
  static_assert(PER == 1 || PER == kStatThreads / 32, "a CTA or a warp per slice");
  pdl_launch_dependents();
  pdl_wait();
  constexpr int kThreads = kStatThreads / PER;
  const int r = blockIdx.x, sl = blockIdx.y * PER + threadIdx.x / kThreads, tid = threadIdx.x % kThreads;
  const float *row = logits + (size_t)r * V;
  const float mx = row_max_of(amax[(size_t)r * kAmaxStride]);
  const int per = slice_len(V), i0 = sl * per, i1 = min(V, i0 + per);
  float sum = 0.f;
#pragma unroll 4
  for (int i = i0 + 4 * tid; i < i1; i += 4 * kThreads) {
    const float4 w = weights4(row, i, mx, inv_t);
    sum += (w.x + w.y) + (w.z + w.w);
  }
  sum = PER == 1 ? cta_sum(sum, red) : warp_sum(sum);
  if (tid == 0) part[(size_t)r * kStatSlices + sl] = sum;
}

// grid = sequences.  The chunk is a draft tree (a chain is the tree with parents j - 1).  Thread c < k computes the
// weight of node c's token under its parent's row; thread 0 then walks from the root: the children of a node are
// tried in node order against the residual (the parent's weights with the tokens of refused children removed),
// child c accepted iff uni[c] * residual total < its weight.  Where the walk ends the block draws the step's one
// sample from the residual with uni[root]: the refused tokens' logits are set to -inf for the draw (their slices' sums are
// taken again) and put back afterwards.  The running sum goes slice by slice over the sums the statistics kernel left,
// and through the one slice in which it passes the target id by id: only that slice of the row is read again (reading the
// whole row twice with one CTA took 39 us of a step on 128 256 ids, this 14).
__global__ void __launch_bounds__(kSampleThreads)
sample_accept_kernel(SampleArgs a) {
  __shared__ float red[kSampleThreads / 32], slice_sum[kStatSlices], warp_tot[kSampleThreads / 32];
  __shared__ float w_node[64], tot_node[64];
  __shared__ int refused[64];
  __shared__ float refused_logit[64];
  __shared__ int sh_l, sh_last, sh_nref, sh_tok, sh_lastw;
  pdl_launch_dependents();
  pdl_wait();
  const int seq = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int r0 = a.in.cu_rows[seq], k = a.in.cu_rows[seq + 1] - r0;
  int32_t *path = a.path + (size_t)seq * a.k_max;
  for (int r = r0 + threadIdx.x; r < r0 + k; r += blockDim.x)
    a.argmax[r] = (int32_t)(0xFFFFFFFFu - (uint32_t)(a.amax[(size_t)r * kAmaxStride] & 0xFFFFFFFFull));
  for (int c = warp; c < k; c += kSampleThreads / 32) {
    const float tot = warp_sum(a.part[(size_t)(r0 + c) * kStatSlices + lane]);   // total weight of node c's own row
    if (lane == 0) tot_node[c] = tot;
  }
  if ((int)threadIdx.x < k) {
    const int c = threadIdx.x, par = a.in.parent[r0 + c];
    w_node[c] = par < 0 ? 0.f
                        : __expf((a.logits[(size_t)(r0 + par) * a.V + a.in.tokens[r0 + c]] - row_max_of(a.amax[(size_t)(r0 + par) * kAmaxStride])) * a.inv_t);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int v = 0, l = 0, nref = 0;
    path[0] = 0;
    for (;;) {
      float R = tot_node[v];
      nref = 0;
      int nxt = -1;
      for (int c = v + 1; c < k; ++c) {
        if (a.in.parent[r0 + c] != v) continue;
        if (a.uni[r0 + c] * R < w_node[c]) { nxt = c; break; }
        R -= w_node[c];
        refused[nref++] = a.in.tokens[r0 + c];
      }
      if (nxt < 0) break;
      v = nxt;
      path[++l] = v;
    }
    sh_l = l; sh_last = v; sh_nref = nref; sh_tok = -1; sh_lastw = -1;
    // the refused tokens leave the row for the draw
    float *row_w = a.logits + (size_t)(r0 + v) * a.V;
    for (int i = 0; i < nref; ++i) { refused_logit[i] = row_w[refused[i]]; row_w[refused[i]] = -INFINITY; }
    __threadfence_block();
  }
  __syncthreads();
  const int l = sh_l, last = sh_last, nref = sh_nref;
  const float *row = a.logits + (size_t)(r0 + last) * a.V;
  const float mx = row_max_of(a.amax[(size_t)(r0 + last) * kAmaxStride]);
  const int per = slice_len(a.V);
  if (threadIdx.x < kStatSlices) slice_sum[threadIdx.x] = a.part[(size_t)(r0 + last) * kStatSlices + threadIdx.x];
  __syncthreads();
  for (int i = 0; i < nref; ++i) {   // (a slice with several refused tokens is taken again for the first of them)
    const int sl = refused[i] / per;
    bool seen = false;
    for (int e = 0; e < i; ++e) seen |= refused[e] / per == sl;
    if (seen) continue;
    float sum = 0.f;
    for (int id = sl * per + 4 * threadIdx.x; id < min(a.V, (sl + 1) * per); id += 4 * kSampleThreads) {
      const float4 w = weights4(row, id, mx, a.inv_t);
      sum += (w.x + w.y) + (w.z + w.w);
    }
    sum = cta_sum(sum, red);
    if (threadIdx.x == 0) slice_sum[sl] = sum;
    __syncthreads();
  }
  float total = 0.f;
  for (int s = 0; s < kStatSlices; ++s) total += slice_sum[s];
  const float target = a.uni[r0] * total;
  // the slice in which the running sum passes the target (none: rounding, or no weight at all)
  float before = 0.f;
  int sl = 0;
  while (sl < kStatSlices && !(before + slice_sum[sl] > target)) before += slice_sum[sl++];
  if (sl < kStatSlices) {
    const int i1 = min(a.V, (sl + 1) * per);
    float run = before;
    bool done = false;
    for (int b0 = sl * per; b0 < i1 && !done; b0 += 4 * kSampleThreads) {   // 2048 ids at a time, four neighbours per thread
      const int id = b0 + 4 * threadIdx.x;
      const float4 w = id < i1 ? weights4(row, id, mx, a.inv_t) : make_float4(0.f, 0.f, 0.f, 0.f);
      const float c0 = w.x, c1 = c0 + w.y, c2 = c1 + w.z, c3 = c2 + w.w;
      float inc = c3;                                  // inclusive prefix over the warp's threads
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const float t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
      }
      __syncthreads();
      if (lane == 31) warp_tot[warp] = inc;
      __syncthreads();
      float base = run, sum = 0.f;
      for (int v = 0; v < kSampleThreads / 32; ++v) {
        if (v < warp) base += warp_tot[v];
        sum += warp_tot[v];
      }
      const float ex = base + (inc - c3);
      // this thread's first id past the target, and the last id that carries weight (the two summation orders may round
      // apart by an ulp: then that one is taken)
      const int hit = (ex + c0 > target && w.x > 0.f) ? id : (ex + c1 > target && w.y > 0.f) ? id + 1
                      : (ex + c2 > target && w.z > 0.f) ? id + 2 : (ex + c3 > target && w.w > 0.f) ? id + 3 : 0x7FFFFFFF;
      const int lw = w.w > 0.f ? id + 3 : w.z > 0.f ? id + 2 : w.y > 0.f ? id + 1 : w.x > 0.f ? id : -1;
      const int first = __reduce_min_sync(0xffffffffu, hit), lastw = __reduce_max_sync(0xffffffffu, lw);
      if (lane == 0) {
        if (first != 0x7FFFFFFF) atomicMin((unsigned int *)&sh_tok, (unsigned int)first);   // (-1 = none yet)
        atomicMax(&sh_lastw, lastw);
      }
      __syncthreads();
      done = sh_tok >= 0;
      run += sum;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int tok = sh_tok >= 0 ? sh_tok : sh_lastw;
    if (tok < 0) {   // rounding kept every partial sum at or below the target: the last id that carries weight
      for (tok = a.V - 1; tok > 0 && !(__expf((row[tok] - mx) * a.inv_t) > 0.f); --tok) {}
    }
    float *row_w = a.logits + (size_t)(r0 + last) * a.V;
    for (int i = 0; i < nref; ++i) row_w[refused[i]] = refused_logit[i];   // the logits are an output: put them back
    int32_t *em = a.emitted + (size_t)seq * a.k_max;
    for (int j = 1; j <= l; ++j) em[j - 1] = a.in.tokens[r0 + path[j]];
    em[l] = tok;
    a.accept_len[seq] = l;
    a.new_len[seq] = a.in.seq_len[seq] + l + 1;
    a.new_pending[seq] = tok;
  }
  __syncthreads();
  publish(a, seq, r0, k, l);
}

template <typename K, typename... Args>
static cudaError_t launch_pdl1(K kernel, dim3 grid, dim3 block, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

cudaError_t launch_sample_accept(const SampleArgs &a, cudaStream_t st) {
  constexpr int kPer = kStatThreads / 32;
  const bool warps = (a.V / 128 + kStatSlices - 1) / kStatSlices * 128 <= kWarpSlice;
  cudaError_t e = launch_pdl1(warps ? row_expsum_kernel<kPer> : row_expsum_kernel<1>, dim3(a.in.M, warps ? kStatSlices / kPer : kStatSlices),
                              dim3(kStatThreads), st, a.logits, a.amax, a.V, a.inv_t, a.part);
  if (e != cudaSuccess) return e;
  return launch_pdl1(sample_accept_kernel, dim3(a.in.B), dim3(kSampleThreads), st, a);
}

}  // namespace ts
