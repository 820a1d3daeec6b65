// Internal interface between the model orchestration (model.cu) and the kernels.
#pragma once
#include <cuda.h>          // CUtensorMap (types only; the driver entry point is resolved at run time)
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "common.cuh"

namespace ts {

// A function attribute (the opt-in to large dynamic shared memory) is set per DEVICE, so "done once" has to be kept
// per device ordinal: bit d of the mask = done on device d.  Setting an attribute twice is harmless, so a race
// between two threads on their first launch costs a repeated call and nothing else.
struct PerDeviceOnce {
  std::atomic<uint64_t> mask{0};
  // true if the caller still has to do the set-up on the current device; *dev receives its ordinal (-1 = unknown)
  bool needed(int *dev) {
    if (cudaGetDevice(dev) != cudaSuccess || *dev < 0 || *dev >= 64) { *dev = -1; return true; }
    return !((mask.load(std::memory_order_acquire) >> *dev) & 1ull);
  }
  void done(int dev) { if (dev >= 0) mask.fetch_or(1ull << dev, std::memory_order_release); }
};

// Per-step inputs resident in device memory (all int32).
struct StepIn {
  const int32_t *tokens;     // [M] chunk ids, rows of sequence i at cu_rows[i]..cu_rows[i+1]
  const int32_t *pos;        // [M] absolute (rotary) position of each row
  const int32_t *slot;       // [M] cache slot the row's K/V go to: cached length + the row's index in its chunk (equal
                             // to pos in a chain; in a draft tree pos is the depth and siblings need slots of their own)
  const int32_t *row_seq;    // [M] sequence index of each row
  const int32_t *cu_rows;    // [B+1]
  const int32_t *seq_len;    // [B] tokens already in the cache
  const int32_t *block_tab;  // [B][pages_per_seq] page ids
  const int32_t *parent;     // [M] parent of each row inside its chunk (row index relative to the chunk; -1 = root)
  const uint32_t *anc;       // [M][2] low / high word of the row's visibility mask over its chunk: bit i = row i of
                             // the chunk is the row itself or one of its ancestors (a chain: bits 0..j)
  const int32_t *row_tile;   // [M] 64 x (first attention tile of the row's sequence) + the row's index in its chunk
  int pages_per_seq;         // (0: all sequences of the step share one row of the block table, as the pieces of a prompt do)
  int B, M;
  BoundsCheck ck;            // ranges for the debug build's index checks
};

// What a projection does with its sums.  EPI_PARTIAL (many-rows kernel): split-K slabs for the next kernel to fold.
// EPI_QKV and EPI_RESID (weight-streaming kernel): the sums are complete inside a thread-block cluster; QKV rotates, stores
// the queries and appends K/V; RESID (O, down) adds to the residual stream and prepares the next projection's input.
enum : int { EPI_PARTIAL = 0, EPI_SWIGLU = 1, EPI_LOGITS = 2, EPI_QKV = 3, EPI_RESID = 4 };

// A row's packed maximum (EPI_LOGITS) has a line of its own: with the rows' words side by side the LM head's thousand atomics
// per row all went to a few lines of L2, one after the other at about 1 ns each: the launch grew by 0.45 us per row.
constexpr int kAmaxStride = 16;   // 128 bytes
struct GemmArgs {
  int N, K, M;          // output features, reduction length, valid activation rows
  int Mc;               // activation rows per CTA: the step's rows rounded up (weight-streaming kernel), 128 (many rows)
  int planes;           // 1 = bf16 activations, 2 = (hi, lo) pair
  int n_kblocks;        // K / 64
  int stages;           // filled in by the launcher
  // many-rows kernel, filled in by the launcher: weight tiles of 256 rows (the tiles after them have 128), narrow tiles of the
  // CTAs with one wide tile less, row chunks, K slices
  int n_wide, narrow_short, chunks, n_splits;
  float *out;           // EPI_PARTIAL: [splits][out_rows][N]; EPI_LOGITS: [M][N]
  int out_rows;
  __nv_bfloat16 *act_out;  // EPI_SWIGLU: [out_planes][act_rows][N/2]
  int act_rows;
  int out_planes;
  unsigned long long *amax;  // EPI_LOGITS: [M][kAmaxStride] packed (ordered logit bits << 32 | ~token id), atomicMax
  int *err;             // device status word
  unsigned long long *stamp;   // optional clock stamps of this launch (null = none)
  // ---- weight-streaming kernel only ----
  // The RMS norm is split between two projections: the one before stores x * gain (not normalised) and, per row and
  // 128-feature tile, the sum of x squared; the one after multiplies its finished sums by rsqrt(mean + eps).
  const float *ss;      // QKV, SWIGLU: [M][ss_tiles] sums of squares of this input's rows; null: the input is normalised
  int ss_tiles;
  float inv_d, eps;
  float *x;             // RESID: [M][N] residual stream, updated in place
  const float *gain;    // RESID: gain of the norm that follows
  __nv_bfloat16 *h_out; // RESID: [out_planes][act_rows][N] x * gain; null: not wanted
  float *ss_out;        // RESID: [M][N / 128]
  StepIn in;            // QKV
  const float2 *rope_tab;
  __half *q_out, *q_lo_out, *k_pages, *v_pages;
  int Hq, Hkv, hd;
};

int gemm_pick_stages(int planes, int Mc, size_t smem_budget);
// clusters of this many CTAs that are resident at once on the current device, at this much shared memory per CTA
int gemm_max_clusters(int cluster, size_t smem_budget);
// cluster: CTAs along K that complete a tile's sums together (QKV, RESID; 1 for the others)
cudaError_t launch_gemm(int epi, const CUtensorMap &tw, const CUtensorMap &ta, GemmArgs g, int cluster,
                        size_t smem_budget, cudaStream_t st, bool pdl);

// The same projections for many rows (gemm_rows_tcgen05.cu): 128 activation rows x 256 weight rows per CTA, one CTA
// per SM.  `ta` must be the activation map whose box holds 128 rows; g.Mc and g.stages are set by the launcher.
int gemm_rows_tiles(int N);
cudaError_t launch_gemm_rows(int epi, const CUtensorMap &tw, const CUtensorMap &ta, GemmArgs g, int n_splits,
                             size_t smem_limit, int n_sms, cudaStream_t st, bool pdl);

// x[m] = E[tokens[m]]; h = rmsnorm(x) * gain -> bf16 (hi[, lo])
cudaError_t launch_embed_norm(const StepIn &in, const __nv_bfloat16 *embed, const float *gain, float eps,
                              int d, float *x, __nv_bfloat16 *h, int h_rows, int planes,
                              unsigned long long *amax, cudaStream_t st);
// x[m] += sum_s part[s][m]; h = rmsnorm(x) * gain -> bf16 (hi[, lo])
cudaError_t launch_add_norm(int M, int d, const float *part, int n_splits, int part_rows, const float *gain,
                            float eps, float *x, __nv_bfloat16 *h, int h_rows, int planes, cudaStream_t st,
                            unsigned long long *stamp = nullptr);
// qkv = sum of split-K partials; rotary on q and k; q -> fp16 [M][Hq][hd] and the rounding remainder of
// every element as a second array of the same shape; k, v -> fp16 pages
cudaError_t launch_rope_kv(const StepIn &in, const float *part, int n_splits, int part_rows, int Hq, int Hkv,
                           int hd, const float2 *rope_tab, __half *q_out, __half *q_lo_out, __half *k_pages,
                           __half *v_pages, cudaStream_t st, unsigned long long *stamp = nullptr);

constexpr int kAttnMaxSplits = 32;   // KV splits per (row tile, kv head): one lane of the merge kernel each

struct AttnArgs {
  StepIn in;
  const __half *q;               // [M][Hq][hd] rotated queries, fp16
  const __half *k_pages;         // [page][Hkv][16][hd], fp16
  const __half *v_pages;
  int Hq, Hkv, hd;
  int n_splits;                  // KV splits per (sequence, kv head, row tile)
  int n_row_tiles_total;         // sum over sequences of row tiles
  const int32_t *tile_seq;       // [n_row_tiles_total] sequence of each row tile
  const int32_t *tile_row0;      // [n_row_tiles_total] first packed row (j*G+g index) of the tile
  float *part_o;                 // [M*Hq][n_splits][hd] unnormalised partial outputs
  float2 *part_ml;               // [M*Hq][n_splits] (running max in log2 domain, sum)
  __nv_bfloat16 *out;            // [planes][out_rows][Hq*hd]
  int out_rows, planes;
};
cudaError_t launch_attention_split(const AttnArgs &a, cudaStream_t st);
cudaError_t launch_attention_combine(const AttnArgs &a, cudaStream_t st);

// tcgen05 attention as a kernel of its own (attention_tc.cu).  A unit of work is (128-row tile of packed rows, kv head,
// run of KV positions); the host lists each CTA's units.  Every unit yields one partial result per row in a slot of its
// own, and the merge adds a row's slots in order of position.
struct AttnWork {
  int32_t seq, r_beg;         // sequence, its first row in the step
  int32_t row0, rows;         // first packed row (chunk row x group + query head of the group) of the tile, rows in it
  int32_t kh_slot;            // kv head | slot << 16
  int32_t pos_beg, pos_end;   // positions (pos_beg is a multiple of 64; an empty run writes an empty slot)
  int32_t len;                // cached length of the sequence: every row sees every position below it
};
struct AttnTcArgs {
  StepIn in;
  int Hq, Hkv, hd, layer;
  int n_ctas;                    // CTA c walks units cta_unit[c] .. cta_unit[c + 1]
  int n_slots;                   // partial results kept per (row, query head): the most units any (tile, kv head) has
  int ready_len;                 // >= 0: positions below it were cached before this step (a step over pieces of one prompt,
                                 // whose `len`s lie inside the step); -1: those below each sequence's own `len` were
  const AttnWork *units;
  const int32_t *cta_unit;
  const int32_t *tile_slots;     // [tiles][Hkv] units of each (tile, kv head)
  const __half *q, *q_lo;        // [M][Hq][hd] rotated queries as an fp16 pair: value and rounding remainder
  const CUtensorMap *map_kv;     // device copy of the 5-d map over the paged KV pool
  float *attn_o;                 // [M*Hq][n_slots][hd] unnormalised partial outputs
  float2 *attn_ml;               // [M*Hq][n_slots] (reference maximum in the log2 domain, sum)
  __nv_bfloat16 *out;            // [planes][out_rows][Hq*hd] merged, normalised rows as bf16 (hi[, lo])
  int out_rows, planes;
  int *err;                      // device status word
  unsigned long long *stamp, *stamp_merge;   // optional clock stamps of the attention and the merge launch
};
cudaError_t launch_attention_tc(const AttnTcArgs &a, cudaStream_t st);
cudaError_t launch_attention_tc_merge(const AttnTcArgs &a, cudaStream_t st);

// A step's results straight to the host: the acceptance kernels write the words of the result block that the host reads to
// pinned memory as well, so that no copy follows them (base: the block on the device, host: the same block as the device
// sees the pinned one; host null: not wanted).  done: a word per sequence in the pinned block that takes the call's number when
// the sequence's results are there (null: the host waits for the stream instead).
struct HostOut {
  const int32_t *base;
  int32_t *host;
  const int *err;   // status word, published too
  int32_t *done;
  int32_t number;
};

// per-row argmax over the LM-head tiles, longest accepted prefix per sequence, new lengths
struct AcceptArgs {
  StepIn in;
  const unsigned long long *amax;   // [M][kAmaxStride] packed per-row maxima written by the LM-head epilogue
  int32_t *argmax;         // [M]
  int32_t *accept_len;     // [B]
  int32_t *emitted;        // [B][k_max]
  int32_t *new_len;        // [B]  cache length after the commit
  int32_t *new_pending;    // [B]
  int32_t *path;           // [B][k_max] chunk rows of the accepted path, root first (accept_len + 1 entries)
  int k_max;
  HostOut ho;
};
cudaError_t launch_accept(const AcceptArgs &a, cudaStream_t st);

constexpr int kSampleSlices = 32;   // slices of a row whose sums of weights are kept
// Speculative-sampling acceptance (sampling.cu): per-row softmax statistics, accept tests, the step's one sample.
struct SampleArgs {
  StepIn in;
  float *logits;                    // [M][V] (refused tokens are masked for the draw and restored)
  const unsigned long long *amax;   // [M][kAmaxStride] packed per-row maxima (argmax is still reported)
  const float *uni;                 // [M] uniforms in [0, 1): row c of a chunk decides node c, the root row's draws the sample
  float *part;                      // [M][kSampleSlices] scratch: per-slice sums of exp((l - max) / T)
  int V;
  float inv_t;                      // 1 / temperature
  int32_t *argmax, *accept_len, *emitted, *new_len, *new_pending, *path;
  int k_max;
  HostOut ho;
};
cudaError_t launch_sample_accept(const SampleArgs &a, cudaStream_t st);

#ifdef __CUDACC__
// tells the host that what the CTA wrote (before a barrier), and all kernels that it waited for, can be read
__device__ __forceinline__ void raise_flag(int32_t *flag, int32_t number) {
  __threadfence_system();
  *reinterpret_cast<volatile int32_t *>(flag) = number;
}

// the results of sequence `seq` (rows r0 .. r0 + k, accepted length l) by the whole CTA, after a barrier
template <typename Args>
__device__ __forceinline__ void publish(const Args &a, int seq, int r0, int k, int l) {
  if (!a.ho.host) return;
  auto put = [&](const int32_t *p) { a.ho.host[p - a.ho.base] = *p; };
  for (int i = threadIdx.x; i < k; i += blockDim.x) put(a.argmax + r0 + i);
  for (int i = threadIdx.x; i <= l; i += blockDim.x) {
    put(a.emitted + (size_t)seq * a.k_max + i);
    put(a.path + (size_t)seq * a.k_max + i);
  }
  if (threadIdx.x == 0) {
    put(a.accept_len + seq);
    put(a.new_len + seq);
    put(a.new_pending + seq);
    if (seq == 0) put(a.ho.err);
  }
  if (!a.ho.done) return;
  __syncthreads();
  if (threadIdx.x == 0) raise_flag(a.ho.done + seq, a.ho.number);
}
#endif

// Rows' Top-K straight to the host, in pinned memory as the device sees it (null: not wanted).  ends: one row, the last kernel of
// a call: behind kTopMax pairs the status word and a word that takes the call's number when all of it is there.
constexpr int kTopMax = 64;
struct PairsOut {
  float *host;
  int32_t number;
  bool ends;
};

// Cosine Top-K over datastore hidden states (retrieval.cu).  scores: [N + 2K] floats; the result pairs (index as int
// bits, score), best first, follow the N scores.  The query is q_dev (fp32 [d]) or, if null, bf16 planes of a row.
cudaError_t launch_topk_cosine(const __nv_bfloat16 *H, int N, int d, const float *q_dev, const __nv_bfloat16 *q_planes,
                               int plane_stride, int planes, int K, float *scores, int n_sms, PairsOut po, int *err, cudaStream_t st);

// Row-wise Top-K (topk.cu): out[r][j] = (column as int bits, value) of the j-th largest entry of row r, lowest column
// on ties.  cand: scratch of n_rows * ceil(n_cols / 4096) * K pairs.
// err is published with po where that ends the call.
cudaError_t launch_topk_rows(const float *x, int n_rows, int n_cols, int K, float2 *cand, float *out, PairsOut po,
                             const int *err, cudaStream_t st);

// After a tree step: move the K/V rows of the accepted path to consecutive cache positions len, len+1, ...
struct CompactArgs {
  StepIn in;
  const int32_t *accept_len;   // [B]
  const int32_t *path;         // [B][k_max]
  int k_max;
  __half *kv_pool;             // layer l: K pages at kv_pool + l * layer_stride, V pages v_offset further
  uint64_t layer_stride, v_offset;
  int n_layers, Hkv, hd;
};
cudaError_t launch_kv_compact(const CompactArgs &a, cudaStream_t st);

// Where a source row of an uploaded matrix goes in the stored matrix: row r -> base + r * mul, or, with
// hd != 0, base + (r / hd) * hd + p(r % hd) with p(e) = 2e for e < hd/2 and 2(e - hd/2) + 1 otherwise.
struct RowMap { int base, mul, hd, tiles; };   // tiles = 128-row blocks of the whole stored matrix
// Index of block (128-row tile, 64-wide k-block) of a stored projection matrix, in units of 128 x 64 blocks: k-block
// major, so that the CTAs of one launch, which walk the k-blocks of neighbouring tiles in step, read one contiguous
// region of memory at a time instead of as many regions a tile's length apart as there are CTAs.
__host__ __device__ inline int w_block(int tile, int kb, int tiles, int kblocks) { (void)kblocks; return kb * tiles + tile; }
// Scatter n_rows source rows (row-major, K columns, first one being row r0 of the uploaded matrix) into the
// 128 x 64-block storage of the stored matrix.
cudaError_t launch_retile(const __nv_bfloat16 *src, int n_rows, int r0, int K, RowMap rm, __nv_bfloat16 *dst,
                          cudaStream_t st);

// ---- fused single-kernel step (fused.cu) ---------------------------------------------------------------
struct FusedArgs {
  // model shape
  int n_layers, d, Nqkv, Nq, F, V, Hq, Hkv, hd;
  float eps;
  // step
  StepIn in;
  int Mc, mc_index, planes;      // activation rows per MMA (16, 32 or 64), its index, 1 or 2 planes
  int n_ctas, ring, attn_smem_bytes, skip_lm, k_max;
  int n_attn_tiles, attn_splits;
  const int32_t *tile_seq;       // [n_attn_tiles] sequence of each 128-row tile of packed rows
  const int32_t *tile_row0;      // [n_attn_tiles] first packed row of the tile
  // tensor maps in device memory: 4 per layer (qkv, o, gate-up, down), LM head, then per row-chunk
  // size three activation maps (h, attn, act)
  const CUtensorMap *maps;
  int map_kv;                    // index of the 5-d map over the paged KV pool (64 elements x 16 positions x head x page x layer*2)
  const __nv_bfloat16 *embed;
  const float *gains;            // g1[0], g2[0], g1[1], ..., gf; gain_stride floats apart
  int gain_stride;
  const float2 *rope;
  __half *kv_pool;
  unsigned long long kv_layer_stride, kv_v_offset;   // in fp16 elements
  // workspace
  float *x;                      // [R][d] residual stream
  __nv_bfloat16 *h, *attn, *act; // [planes][R][.]
  int R;
  __half *q;                     // [R][Hq*hd]
  float *slab;                   // [n_ctas][2][Mc][128] parked partial tiles
  float *ss_part;                // [d/128][R] per-tile sums of squares of x
  float *attn_o;                 // [M*Hq][splits][hd]
  float2 *attn_ml;               // [M*Hq][splits]
  float *logits;                 // [M][V]
  unsigned long long *amax;      // [M]
  int *sync;                     // [0] phase counter, [2] exit counter, [8..] tile counters (all zero between launches)
  int *err;                      // device status word shared with the other kernels
  int n_counters;
  // optional clocks (ns, latest over the CTAs), three rows of n_phases: phase end; last MMA of the phase
  // issued; first weight+activation block of the phase ready
  unsigned long long *phase_t;
  int n_phases;
  // results
  int32_t *out_argmax, *out_accept, *out_emitted, *out_newlen, *out_newpend;
};
size_t fused_attn_smem_bytes(int hd);
int fused_ring_stages(int planes, int Mc, int hd, size_t smem_limit);
cudaError_t launch_fused(FusedArgs a, size_t smem_limit, cudaStream_t st);

}  // namespace ts
