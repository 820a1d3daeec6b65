// The dense projections of the verify step for MANY rows (batched steps and prompts: more than the weight-streaming kernel
// takes, 80 rows or 96 with one plane of activations), where the work is bound by
// the tensor cores and by the bytes an SM pulls from L2 per flop, no longer by streaming the weights:
//     out[m][n] = sum_k act[m][k] * W[n][k]
// Orientation: a CTA owns a chunk of 128 activation rows (operand A of the tensor-core instruction, its 128-row
// dimension) and 256 weight rows (operand B, the instruction's N dimension); the accumulator in tensor memory is
// 128 lanes (rows) x 256 fp32 columns (features).  The (hi, lo) bf16 planes of the activations are two instructions
// into the SAME accumulator, so per 64-wide k-block a CTA brings in 32 KB of activations and 32 KB of weights for
// 8.4 MFLOP -- two thirds of the bytes per flop of the weight-streaming kernel (gemm_tcgen05.cu), which at these sizes
// is what sets the pace.  The weight matrix keeps its storage (contiguous 128 x 64 blocks, one TMA box each): a CTA's
// 256 weight rows are two such boxes.  One CTA per SM (three 64 KB stages), and the launch has no more CTAs than SMs: a CTA
// walks its tiles one after the other with two accumulators in tensor memory, so that the loads of the next tile and its
// products run under the epilogue of this one.  (A CTA per tile paid 8 to 10 us for set-up, first loads and epilogue each
// time, against 40 of main loop for the longest tiles; 1024 rows of the 8B shape: gate-up 328 -> 300 us, 1.37 PFLOP/s of issued
// work, the rate a sustained cuBLAS product reaches under the power cap.)
//
// Roles: warp 0 = TMA producer, warp 1 = TMEM allocation + MMA issue, warps 2..9 = epilogue (thread <-> row, two
// warps per row quarter, half of the columns each).
// Every wait is bounded; on expiry the CTA records an error word and leaves through the normal exit.
#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

#include "kernels.h"

namespace ts {

static constexpr int kBlockK = 64;                 // k-block: 64 bf16 = 128 bytes per row
static constexpr int kRowsM = 128;                 // activation rows per CTA
static constexpr int kBoxN = 128;                  // weight rows per stored block (one TMA box)
static constexpr int kTileN = 256;                 // weight rows per CTA
static constexpr int kBoxBytes = kBoxN * kBlockK * 2;
static constexpr int kMaxStages = 4;

struct __align__(8) RowsSmemCtl {
  uint64_t full[kMaxStages];
  uint64_t empty[kMaxStages];
  uint64_t acc_full[2];    // [accumulator]
  uint64_t acc_empty[2];
  uint32_t tmem_base;
  uint32_t abort_flag;
};
static constexpr int kStagingBytes = 8 * 4096;   // per epilogue warp 32 rows x 128 bytes

// One output tile of a launch: rows [m0, m0 + 128), stored weight blocks blk0 (and blk0 + 1 if nb = 256), k-blocks [kb0, kb1).
struct RowsTile {
  int m0, blk0, nb, split, kb0, nkb;
};
// The tiles of CTA c out of G.  Wide tiles (two weight blocks) are dealt out in turn; of the narrow ones the first
// g.narrow_short go in turn to the CTAs that got one wide tile less (all of them, if it came out even), the others to the
// rest: the launcher has chosen the counts.  Row chunks are neighbours in the order: they run at the same time and all but
// the first find the weight blocks in L2.
struct RowsShare {   // of this CTA: its wide tiles, then the narrow ones first, first + step, .. below end
  int wides, first, step, end;
};
__device__ __forceinline__ RowsShare rows_share(const GemmArgs &g, int c, int G) {
  const int nW = g.n_wide * g.chunks * g.n_splits, nN = (g.N / kBoxN - 2 * g.n_wide) * g.chunks * g.n_splits;
  const int q = nW / G, r = nW - q * G;
  return c < r ? RowsShare{q + 1, g.narrow_short + c, r, nN} : RowsShare{q, c - r, G - r, g.narrow_short};
}
// j = how many tiles this CTA has had; false: no more.  (Few and 32-bit divisions: every role of a CTA goes through this
// before its first tile and once more after its last.  With two of 64 bits and the share worked out each time a launch of one
// tile per CTA took 0.5 to 1 us more; steps of 128 rows 186.2 -> 184.4 us on two 1B layers, 308 -> 304 on two 8B ones.)
__device__ __forceinline__ bool rows_tile(const GemmArgs &g, const RowsShare &p, int c, int G, int j, RowsTile &t) {
  const bool wide = j < p.wides;
  const int u = wide ? c + j * G : p.first + (j - p.wides) * p.step;
  if (!wide && u >= p.end) return false;
  t.nb = wide ? kTileN : kBoxN;
  const int v = g.chunks == 1 ? u : u / g.chunks;
  t.m0 = (u - v * g.chunks) * kRowsM;
  int tile = v;
  t.split = t.kb0 = 0;
  t.nkb = g.n_kblocks;
  if (g.n_splits > 1) {
    const int n_tiles = wide ? g.n_wide : g.N / kBoxN - 2 * g.n_wide;
    t.split = v / n_tiles;
    tile = v - t.split * n_tiles;
    t.kb0 = t.split * g.n_kblocks / g.n_splits;   // balanced cut of the k-blocks
    t.nkb = (t.split + 1) * g.n_kblocks / g.n_splits - t.kb0;
  }
  t.blk0 = wide ? 2 * tile : 2 * g.n_wide + tile;
  return true;
}

template <int EPI>
__global__ void __launch_bounds__(320, 1)
gemm_rows_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_a,
                 const GemmArgs g) {
  extern __shared__ uint8_t smem_raw[];
  // 1024-byte alignment is required by the 128-byte swizzle pattern
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int a_bytes = g.planes * kRowsM * kBlockK * 2;
  const int stage_bytes = a_bytes + 2 * kBoxBytes;
  uint8_t *staging = smem + (size_t)g.stages * stage_bytes;
  RowsSmemCtl *ctl = reinterpret_cast<RowsSmemCtl *>(staging + kStagingBytes);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cta = blockIdx.x, G = gridDim.x;
  const RowsShare share = rows_share(g, cta, G);

  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&tmap_w);
    tma_prefetch_desc(&tmap_a);
    for (int s = 0; s < g.stages; ++s) {
      mbar_init(smem_u32(&ctl->full[s]), 1);
      mbar_init(smem_u32(&ctl->empty[s]), 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(smem_u32(&ctl->acc_full[s]), 1);
      mbar_init(smem_u32(&ctl->acc_empty[s]), 8);   // one arrival per epilogue warp
    }
    ctl->abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&ctl->tmem_base), 2 * kTileN);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = ctl->tmem_base;
  if (threadIdx.x == 0) stamp_min(g.stamp);
  // (placed after this CTA holds its resources, so a waiting dependent can never starve an earlier kernel)
  pdl_launch_dependents();

  if (warp == 0) {
    // ------------------------------------------------------------------ producer
    if (lane == 0) {
      const uint64_t pol_w = policy_evict_first(), pol_a = policy_evict_last();
      // block (128-row block j, k-block kb) of the stored matrix = rows w_block(j, kb) * 128 .. of a [.][64] array
      auto load_w = [&](const RowsTile &t, int s, int kb) {
        const uint32_t bar = smem_u32(&ctl->full[s]);
        const uint32_t dst = smem_u32(smem + (size_t)s * stage_bytes + a_bytes);
        mbar_expect_tx(bar, a_bytes + (t.nb / kBoxN) * kBoxBytes);
        for (int j = 0; j < t.nb / kBoxN; ++j)
          tma_load_2d(dst + j * kBoxBytes, &tmap_w, 0, w_block(t.blk0 + j, kb, g.N / kBoxN, g.n_kblocks) * kBoxN, bar, pol_w);
      };
      auto load_a = [&](const RowsTile &t, int s, int kb) {
        tma_load_3d(smem_u32(smem + (size_t)s * stage_bytes), &tmap_a, kb * kBlockK, t.m0, 0, smem_u32(&ctl->full[s]), pol_a);
      };
      RowsTile t;
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int j = 0; ok && rows_tile(g, share, cta, G, j, t); ++j) {
        int it = 0;
        if (j == 0) {
          // weights do not depend on the previous kernel: start them before the programmatic-dependency wait
          const int pre = min(g.stages, t.nkb);
          for (int i = 0; i < pre; ++i) load_w(t, i, t.kb0 + i);
          pdl_wait();
          stamp_waited(g.stamp);
          for (int i = 0; i < pre; ++i) load_a(t, i, t.kb0 + i);
          it = pre;
          s = pre == g.stages ? 0 : pre;
          ph = pre == g.stages ? 1 : 0;
        }
        for (; it < t.nkb; ++it) {
          if (!mbar_wait(smem_u32(&ctl->empty[s]), ph ^ 1)) {
            atomicExch(g.err, DEV_TIMEOUT_EMPTY);
            ok = false;
            break;
          }
          load_w(t, s, t.kb0 + it);
          load_a(t, s, t.kb0 + it);
          if (++s == g.stages) { s = 0; ph ^= 1; }
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issue
    // The whole warp walks the loop and the waits; one elected lane issues the instructions of a k-block and its commit.
    RowsTile t;
    int s = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int j = 0; ok && rows_tile(g, share, cta, G, j, t); ++j) {
      const int b = j & 1;
      const uint32_t idesc = umma_idesc_bf16(kRowsM, (uint32_t)t.nb), d = tmem_base + b * kTileN;
      // the accumulator's previous tile has been read out
      if (j >= 2 && !__all_sync(0xffffffffu, mbar_wait(smem_u32(&ctl->acc_empty[b]), ((j >> 1) - 1) & 1))) {
        if (lane == 0) atomicExch(g.err, DEV_TIMEOUT_TMEM);
        ok = false;
      }
      for (int it = 0; ok && it < t.nkb; ++it) {
        if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&ctl->full[s]), ph))) {   // (all lanes leave together)
          if (lane == 0) atomicExch(g.err, DEV_TIMEOUT_FULL);
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t sa = smem_u32(smem + (size_t)s * stage_bytes);
        const uint64_t db = umma_desc_sw128(sa + a_bytes);
        if (elect_one()) {
          // the value plane and the remainder plane of the activations into the same sums
          for (int pl = 0; pl < g.planes; ++pl) {
            const uint64_t da = umma_desc_sw128(sa + pl * (kRowsM * kBlockK * 2));
#pragma unroll
            for (int kk = 0; kk < kBlockK / 16; ++kk)   // 16 bf16 along K = 32 bytes = 2 descriptor address units
              umma_bf16(d, da + 2 * kk, db + 2 * kk, idesc, (it | kk | pl) != 0);
          }
          umma_commit(smem_u32(&ctl->empty[s]));
        }
        __syncwarp();
        if (++s == g.stages) { s = 0; ph ^= 1; }
      }
      if (elect_one()) {
        if (!ok) *reinterpret_cast<volatile uint32_t *>(&ctl->abort_flag) = 1;
        umma_commit(smem_u32(&ctl->acc_full[b]));
      }
      __syncwarp();
    }
  } else {
    // ------------------------------------------------------------------ epilogue (warps 2..9): thread <-> row
    pdl_wait();   // outputs of this kernel may still be read by the previous one's consumers
    const int q = warp & 3;                       // TMEM lane quarter this warp may read
    const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16);
    // Results leave through shared memory so that global stores are whole lines: a thread owns a ROW of the
    // accumulator, so storing from registers makes the 32 lanes of a warp write 32 different lines per instruction
    // (4 us for the 128 KB of a tile).  Each warp stages 32 rows x 128 bytes (16-byte chunks, slot = chunk ^ (row & 7):
    // conflict-free both ways) in a buffer of its own and writes them back 4 rows x 128 bytes per instruction.
    // Eight epilogue warps: warps 2..5 take the first half of the tile's columns, warps 6..9 the second (two warps
    // per tensor-memory lane quarter).
    const int eh = (warp - 2) >> 2;
    const uint32_t stg = smem_u32(staging) + (warp - 2) * 4096;
    const int rr = lane >> 3, slot = lane & 7;   // read-back: rows rr, rr + 4, ...; 16-byte slot of the row
    RowsTile t;
    for (int j = 0; rows_tile(g, share, cta, G, j, t); ++j) {
      const int b = j & 1;
      bool ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&ctl->acc_full[b]), (j >> 1) & 1));
      if (!ok && lane == 0) atomicExch(g.err, DEV_TIMEOUT_TMEM);
      tc_fence_after();
      ok = ok && (*reinterpret_cast<volatile uint32_t *>(&ctl->abort_flag) == 0);
      if (!ok) break;
      const int m0 = t.m0, n0 = t.blk0 * kBoxN, split = t.split;
      const int m = m0 + q * 32 + lane;             // this thread's row
      const bool row_ok = m < g.M;
      const uint32_t tacc = taddr + b * kTileN;
      float best = -INFINITY;
      int best_n = 0;
      const int c_beg = eh * (t.nb >> 1), c_end = c_beg + (t.nb >> 1);
      // (the sums are out of tensor memory when a warp has read its last columns)
      auto read_done = [&](int c_next) {
        if (c_next < c_end) return;
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&ctl->acc_empty[b]));
      };
      if constexpr (EPI != EPI_SWIGLU) {
        for (int c0 = c_beg; c0 < c_end; c0 += 32) {
          uint32_t r[32];
          tmem_ld16(tacc + c0, *reinterpret_cast<uint32_t(*)[16]>(r));     // (warp-wide: rows past the end read too)
          tmem_ld16(tacc + c0 + 16, *reinterpret_cast<uint32_t(*)[16]>(r + 16));
          tmem_wait_ld();
          read_done(c0 + 32);
          const int n = n0 + c0;
          if constexpr (EPI == EPI_LOGITS) {
            if (row_ok) {
#pragma unroll
              for (int j = 0; j < 32; ++j) {
                const float v = __uint_as_float(r[j]);
                if (v > best) { best = v; best_n = n + j; }   // (ascending ids: a tie keeps the lower one)
              }
            }
          }
#pragma unroll
          for (int c = 0; c < 8; ++c)
            st_shared_v4(stg + lane * 128 + ((c ^ (lane & 7)) << 4), r[4 * c], r[4 * c + 1], r[4 * c + 2], r[4 * c + 3]);
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int R = i * 4 + rr, mr = m0 + q * 32 + R;
            const uint4 v = ld_shared_v4(stg + R * 128 + ((slot ^ (R & 7)) << 4));
            if (mr < g.M) {
              float *dst = (EPI == EPI_PARTIAL ? g.out + ((size_t)split * g.out_rows + mr) * g.N : g.out + (size_t)mr * g.N) + n + slot * 4;
              *reinterpret_cast<uint4 *>(dst) = v;
            }
          }
          __syncwarp();
        }
      } else {
        // EPI_SWIGLU: even feature = gate_f, odd = up_f, f = n / 2.  64 accumulator columns give 32 features: 64 bytes
        // of the value plane (slots 0..3 of the staged row) and 64 of the remainder plane (slots 4..7).
        const int F = g.N >> 1;
        for (int c0 = c_beg; c0 < c_end; c0 += 64) {
          uint32_t hi[16], lo[16];   // 32 features per plane, two bf16 per word
#pragma unroll
          for (int part = 0; part < 4; ++part) {
            uint32_t r[16];
            tmem_ld16(tacc + c0 + part * 16, r);
            tmem_wait_ld();
            if (part == 3) read_done(c0 + 64);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              __nv_bfloat16 h0, l0, h1, l1;
              const float g0 = __uint_as_float(r[4 * j]), u0 = __uint_as_float(r[4 * j + 1]);
              const float g1 = __uint_as_float(r[4 * j + 2]), u1 = __uint_as_float(r[4 * j + 3]);
              split_bf16(g0 / (1.f + __expf(-g0)) * u0, h0, l0);
              split_bf16(g1 / (1.f + __expf(-g1)) * u1, h1, l1);
              hi[part * 4 + j] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
              lo[part * 4 + j] = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
            }
          }
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            st_shared_v4(stg + lane * 128 + ((c ^ (lane & 7)) << 4), hi[4 * c], hi[4 * c + 1], hi[4 * c + 2], hi[4 * c + 3]);
            st_shared_v4(stg + lane * 128 + (((c + 4) ^ (lane & 7)) << 4), lo[4 * c], lo[4 * c + 1], lo[4 * c + 2], lo[4 * c + 3]);
          }
          __syncwarp();
          const int f = (n0 + c0) >> 1;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int R = i * 4 + rr, mr = m0 + q * 32 + R;
            const uint4 v = ld_shared_v4(stg + R * 128 + ((slot ^ (R & 7)) << 4));
            if (mr < g.M && (slot < 4 || g.out_planes == 2)) {
              __nv_bfloat16 *dst = g.act_out + ((size_t)(slot < 4 ? 0 : g.act_rows) + mr) * F + f + (slot & 3) * 8;
              *reinterpret_cast<uint4 *>(dst) = v;
            }
          }
          __syncwarp();
        }
      }
      if constexpr (EPI == EPI_LOGITS) {
        if (row_ok) {
          // order-preserving map of the float to an unsigned word; ties resolve to the lowest id
          uint32_t u = __float_as_uint(best);
          u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
          atomicMax(g.amax + (size_t)m * kAmaxStride, ((unsigned long long)u << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)best_n));
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 2 * kTileN);
  }
  if (threadIdx.x == 0 && g.stamp) stamp_max(g.stamp + 3);
}

static size_t rows_smem_bytes(int stages, int planes) {
  return (size_t)stages * (planes * kRowsM * kBlockK * 2 + 2 * kBoxBytes) + kStagingBytes + sizeof(RowsSmemCtl) + 1024;
}

template <int EPI>
static cudaError_t launch_rows_one(const CUtensorMap &tw, const CUtensorMap &ta, const GemmArgs &g, dim3 grid,
                                   size_t smem, cudaStream_t st, bool pdl) {
  static PerDeviceOnce once;
  int dev_ = -1;
  if (once.needed(&dev_)) {
    cudaError_t e = cudaFuncSetAttribute(gemm_rows_kernel<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e != cudaSuccess) return e;
    once.done(dev_);
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(320);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, gemm_rows_kernel<EPI>, tw, ta, g);
}

int gemm_rows_tiles(int N) { return (N + kTileN - 1) / kTileN; }

// How a launch's tiles are dealt out (see rows_tile).  A launch that is not cut along K mixes tile widths: a narrow tile
// costs about 0.6 of a wide one (half the flops, three quarters of the bytes through shared memory), and with the last
// tiles narrow the CTAs end closer together.  The count of wide tiles, and how many narrow ones go to the CTAs that have
// one wide tile less, with the earliest finish win; ties go to fewer narrow tiles.
static constexpr double kNarrowCost = 0.6;
struct Deal { int n_wide, narrow_short; };
static Deal pick_deal(int blocks, int chunks, int splits, int G, bool mix) {
  static std::mutex mu;
  static std::map<std::tuple<int, int, int, int, bool>, Deal> memo;   // (a pure function of its key: shapes and SM count)
  std::lock_guard<std::mutex> lk(mu);
  const auto key = std::make_tuple(blocks, chunks, splits, G, mix);
  auto it = memo.find(key);
  if (it != memo.end()) return it->second;
  Deal best{blocks / 2, 0};
  double best_t = 1e30;
  const int x_max = blocks / 2, x_min = mix ? std::max(0, x_max - 2 * G / chunks) : x_max;
  for (int x = x_max; x >= x_min; --x) {
    const int nW = x * chunks * splits, nN = (blocks - 2 * x) * chunks * splits, r = nW % G, S = G - r;
    // ns narrow tiles over S CTAs from the start of the last round, the others over r CTAs one wide tile later
    double t_x = 1e30;
    int ns_x = nN;
    for (int ns = r ? 0 : nN; ns <= nN; ++ns) {
      const double t = std::max(kNarrowCost * ((ns + S - 1) / S), r ? 1.0 + kNarrowCost * ((nN - ns + r - 1) / r) : 0.0);
      if (t < t_x - 1e-9) { t_x = t; ns_x = ns; }
    }
    t_x += nW / G;
    if (t_x < best_t - 1e-9) { best_t = t_x; best = {x, ns_x}; }
  }
  memo[key] = best;
  return best;
}

// `ta` must be the activation map whose box holds 128 rows.  N must be a multiple of 128.
cudaError_t launch_gemm_rows(int epi, const CUtensorMap &tw, const CUtensorMap &ta, GemmArgs g, int n_splits,
                             size_t smem_limit, int n_sms, cudaStream_t st, bool pdl) {
  if (n_splits < 1 || n_splits > g.n_kblocks || g.N % kBoxN) return cudaErrorInvalidValue;
  g.Mc = kRowsM;
  g.stages = kMaxStages;
  while (g.stages > 2 && rows_smem_bytes(g.stages, g.planes) > smem_limit) --g.stages;
  const size_t smem = rows_smem_bytes(g.stages, g.planes);
  if (smem > smem_limit) return cudaErrorInvalidConfiguration;
  const int blocks = g.N / kBoxN;
  g.chunks = (g.M + kRowsM - 1) / kRowsM;
  g.n_splits = n_splits;
  // split-K launches are already cut to fill their rounds; the others may mix tile widths
  const bool mix = n_splits == 1;
  const int G = mix ? n_sms : std::min(n_sms, (blocks + 1) / 2 * g.chunks * n_splits);
  const Deal deal = pick_deal(blocks, g.chunks, n_splits, G, mix);
  g.n_wide = deal.n_wide;
  g.narrow_short = deal.narrow_short;
  dim3 grid(G);
  switch (epi) {
    case EPI_PARTIAL: return launch_rows_one<EPI_PARTIAL>(tw, ta, g, grid, smem, st, pdl);
    case EPI_SWIGLU: return launch_rows_one<EPI_SWIGLU>(tw, ta, g, grid, smem, st, pdl);
    default: return launch_rows_one<EPI_LOGITS>(tw, ta, g, grid, smem, st, pdl);
  }
}

}  // namespace ts
