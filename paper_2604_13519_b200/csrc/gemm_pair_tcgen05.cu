// The dense projections of the verify step for MANY rows by pairs of CTAs:
//     out[m][n] = sum_k act[m][k] * W[n][k]
// A tile is 256 weight rows times a chunk of up to 256 activation rows, worked on by a cluster of two CTAs, one per SM: one
// tensor-core instruction spans both, 128 weight rows of each as its row dimension, half of the activation rows in each one's
// shared memory as the other.  The rows of a step are the N of the instruction, which comes in steps of 16: a step of 144 rows is
// one chunk of 144, where the row-major kernel (gemm_rows_tcgen05.cu) works on two of 128 -- what a step of few more rows than a
// multiple of 128 gains most (8B shape, per layer under the power cap: 144 rows 208 -> 148 us, 192 rows 229 -> 176, 288 rows 283 ->
// 246).  The (hi, lo) bf16 planes of the activations are two instructions into the SAME sums, or, in chunks of up to 128 rows, one
// instruction into sums of their own, added in the epilogue as the weight-streaming kernel adds them.  The sums lie in tensor
// memory, lane = weight row, column = activation row, in two sets: the loads and products of a pair's next tile run under the epilogue of
// this one.  A k-block is 0.64 us at 256 rows (floor 0.52 at 1965 MHz), 0.35 at 144.
//
// The launch is persistent, at most one pair per two SMs.  Every pair has the same number of whole tiles; the tiles that are
// left over are cut along K into equal pieces, dealt out one or more to a pair and worked on FIRST: their sums go to slabs in
// memory, and the CTA that completes a tile adds the slabs in K order, while its pair's products go on with the next tile, and
// finishes the tile.  Nobody waits for another pair.  (Gate-up of the 8B shape at 256 rows: 96 tiles for 74 pairs, 90 -> 79 us
// against the row-major kernel's mix of tile widths.)  EPI_PARTIAL has all of its tiles cut alike and leaves the slabs to the
// next kernel.
//
// Roles: warp 0 = TMA producer (of the CTA's own half), warp 1 = TMEM allocation and, in the pair's first CTA, MMA issue, warps
// 2..9 = epilogue, two groups of four.
// Every wait is bounded; on expiry the CTA records an error word and leaves through the normal exit.
#include <algorithm>

#include "kernels.h"

namespace ts {

static constexpr int kBlockK = 64;                 // k-block: 64 bf16 = 128 bytes per row
static constexpr int kBoxN = 128;                  // weight rows per stored block (one TMA box): a CTA's part of a tile
static constexpr int kBoxBytes = kBoxN * kBlockK * 2;
static constexpr int kMaxStages = 8;

struct __align__(8) PairSmemCtl {
  uint64_t full[kMaxStages];   // (the first CTA's count for both)
  uint64_t empty[kMaxStages];
  uint64_t acc_full[2];        // [set of sums]
  uint64_t acc_empty[2];       // (of the first CTA)
  uint32_t tmem_base;
  uint32_t abort_flag;
  uint32_t last;               // this CTA completed the tile whose slab it wrote last
  float rs[2][128];            // [item in turn][row]: 1 / rms of the input (where it is not normalised yet: g.ss)
};
static constexpr int kFoldAhead = 3;                       // slabs that are read at a time
static constexpr int kPassRows = 16;                       // activation rows that an epilogue group stages at a time
static constexpr int kPassBytes = kPassRows * kBoxN * 4;
static constexpr int kStagingBytes = 2 * 2 * kPassBytes;   // [group][buffer]

// One piece of work of a pair: tile (256 weight rows, chunk), k-blocks [kb0, kb0 + nkb).  cut: the number of the tile among those
// cut along K, -1: a whole tile.
struct PairItem {
  int wt, m0, rows, kb0, nkb, cut, slice;
};
// Item j of pair p out of P; false: no more.  (Neighbours in the order are row chunks of one weight tile: they run at the same
// time and all but the first find the weight blocks in L2.)
__device__ __forceinline__ bool pair_item(const PairArgs &g, int p, int P, int j, PairItem &t) {
  const int n_cut = g.n_tiles - g.n_whole, n_pieces = n_cut * g.pieces;
  const int mine = p < n_pieces ? (n_pieces - 1 - p) / P + 1 : 0;   // pieces of this pair
  int tile;
  if (j < mine) {
    const int u = p + j * P;
    t.slice = u / n_cut;
    t.cut = u - t.slice * n_cut;
    tile = g.n_whole + t.cut;
    t.kb0 = t.slice * g.n_kblocks / g.pieces;   // balanced cut of the k-blocks
    t.nkb = (t.slice + 1) * g.n_kblocks / g.pieces - t.kb0;
  } else {
    tile = p + (j - mine) * P;
    if (tile >= g.n_whole) return false;
    t.cut = -1;
    t.slice = t.kb0 = 0;
    t.nkb = g.n_kblocks;
  }
  t.wt = tile / g.chunks;
  const int c = tile - t.wt * g.chunks;
  t.rows = c < g.n_wide ? g.chunk_rows : g.chunk_rows - 16;
  t.m0 = c * g.chunk_rows - max(0, c - g.n_wide) * 16;
  return true;
}

template <int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(320, 1)
gemm_pair_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_a,
                 const __grid_constant__ CUtensorMap tmap_a_less, const PairArgs g) {
  extern __shared__ uint8_t smem_raw[];
  // 1024-byte alignment is required by the 128-byte swizzle pattern (both CTAs of a pair have the same layout)
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int half_bytes = g.chunk_rows / 2 * kBlockK * 2;   // one plane of this CTA's half of a full chunk
  const int stage_bytes = kBoxBytes + g.planes * half_bytes;
  uint8_t *staging = smem + (size_t)g.stages * stage_bytes;
  PairSmemCtl *ctl = reinterpret_cast<PairSmemCtl *>(staging + kStagingBytes);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_rank(), pair = blockIdx.x >> 1, P = gridDim.x >> 1;
  const int n_blocks = g.N / kBoxN;
  const bool apart = g.planes == 2 && g.chunk_rows <= 128;   // the planes' sums in columns of their own
  const int set_cols = apart ? 2 * g.chunk_rows : g.chunk_rows;
  uint32_t alloc_cols = 32;
  while (alloc_cols < 2u * set_cols) alloc_cols <<= 1;

  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&tmap_w);
    tma_prefetch_desc(&tmap_a);
    tma_prefetch_desc(&tmap_a_less);
    for (int s = 0; s < g.stages; ++s) {
      mbar_init(smem_u32(&ctl->full[s]), 1);
      mbar_init(smem_u32(&ctl->empty[s]), 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(smem_u32(&ctl->acc_full[s]), 1);
      mbar_init(smem_u32(&ctl->acc_empty[s]), 16);   // one arrival per epilogue warp of the pair
    }
    ctl->abort_flag = 0;
    fence_barrier_init();
  }
  __syncwarp();
  if (warp == 1) {
    tmem_alloc_pair(smem_u32(&ctl->tmem_base), alloc_cols);
  }
  tc_fence_before();
  __syncthreads();
  cluster_arrive();   // (both CTAs' barriers are set up before either's loads or products count on them)
  cluster_wait();
  // The permit to allocate is the pair's: it goes back only when both CTAs hold their tensor memory.  (Given back behind the
  // own allocation, it was gone for the CTA that came second, which then waited in its allocation for good: seen after some
  // tens of steps back to back, 60 pairs of QKV of 640 rows, whose CTAs start under the embedding kernel's and so apart.)
  if (warp == 1) tmem_relinquish_pair();
  tc_fence_after();
  const uint32_t tmem_base = ctl->tmem_base;
  if (threadIdx.x == 0) stamp_min(g.stamp);
  // (placed after this CTA holds its resources, so a waiting dependent can never starve an earlier kernel)
  pdl_launch_dependents();

  if (warp == 0) {
    // ------------------------------------------------------------------ producer
    if (lane == 0) {
      const uint64_t pol_w = policy_evict_first(), pol_a = policy_evict_last();
      const uint32_t full0 = cluster_addr(smem_u32(&ctl->full[0]), 0);
      // block (128-row block j, k-block kb) of the stored matrix = rows w_block(j, kb) * 128 .. of a [.][64] array.  (With an odd
      // number of blocks the last tile's second CTA takes the last block once more and writes nothing.)
      auto load_w = [&](const PairItem &t, int s, int kb) {
        if (rank == 0) mbar_expect_tx(smem_u32(&ctl->full[s]), 2u * (kBoxBytes + g.planes * t.rows * kBlockK));
        tma_load_2d_pair(smem_u32(smem + (size_t)s * stage_bytes), &tmap_w, 0,
                         w_block(min(2 * t.wt + rank, n_blocks - 1), kb, n_blocks, g.n_kblocks) * kBoxN, full0 + s * 8, pol_w);
      };
      auto load_a = [&](const PairItem &t, int s, int kb) {
        tma_load_3d_pair(smem_u32(smem + (size_t)s * stage_bytes) + kBoxBytes, t.rows == g.chunk_rows ? &tmap_a : &tmap_a_less,
                         kb * kBlockK, t.m0 + rank * (t.rows / 2), 0, full0 + s * 8, pol_a);
      };
      PairItem t;
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int j = 0; ok && pair_item(g, pair, P, j, t); ++j) {
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
    // ------------------------------------------------------------------ MMA issue (the pair's first CTA)
    // The whole warp walks the loop and the waits; one elected lane issues the instructions of a k-block and its commit.
    PairItem t;
    int s = 0;
    uint32_t ph = 0;
    bool ok = rank == 0;
    for (int j = 0; ok && pair_item(g, pair, P, j, t); ++j) {
      const int b = j & 1;
      // (planes apart: a CTA's half of B is its half of the rows of the value plane, then the same of the remainder plane)
      const uint32_t idesc = umma_idesc_bf16(2 * kBoxN, (uint32_t)(apart ? 2 * t.rows : t.rows)), d = tmem_base + b * set_cols;
      const int instr = apart ? 1 : g.planes;
      const uint32_t lo16 = (uint32_t)(t.rows / 2 * kBlockK * 2) >> 4;   // from the value plane to the remainder plane
      // this set's previous sums have been read out
      if (j >= 2 && !__all_sync(0xffffffffu, mbar_wait_cluster(smem_u32(&ctl->acc_empty[b]), ((j >> 1) - 1) & 1))) {
        if (lane == 0) atomicExch(g.err, DEV_TIMEOUT_TMEM);
        ok = false;
      }
      tc_fence_after();
      for (int it = 0; ok && it < t.nkb; ++it) {
        if (!__all_sync(0xffffffffu, mbar_wait_cluster(smem_u32(&ctl->full[s]), ph))) {   // (all lanes leave together)
          if (lane == 0) atomicExch(g.err, DEV_TIMEOUT_FULL);
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t sa = smem_u32(smem + (size_t)s * stage_bytes);
        const uint64_t da = umma_desc_sw128(sa), db = umma_desc_sw128(sa + kBoxBytes);
        if (elect_one()) {
          // the value plane and the remainder plane of the activations into the same sums
          for (int pl = 0; pl < instr; ++pl) {
#pragma unroll
            for (int kk = 0; kk < kBlockK / 16; ++kk)   // 16 bf16 along K = 32 bytes = 2 descriptor address units
              umma_bf16_pair(d, da + 2 * kk, db + pl * lo16 + 2 * kk, idesc, (it | kk | pl) != 0);
          }
          umma_commit_pair(smem_u32(&ctl->empty[s]));
        }
        __syncwarp();
        if (++s == g.stages) { s = 0; ph ^= 1; }
      }
      if (elect_one()) {
        if (!ok) {
          st_cluster_u32(cluster_addr(smem_u32(&ctl->abort_flag), 0), 1);
          st_cluster_u32(cluster_addr(smem_u32(&ctl->abort_flag), 1), 1);
        }
        umma_commit_pair(smem_u32(&ctl->acc_full[b]));
      }
      __syncwarp();
    }
  } else {
    // ------------------------------------------------------------------ epilogue (warps 2..9)
    // Two groups of four warps take the columns (activation rows) sixteen at a time in turn.  First thread <-> weight row: a
    // group's columns go to shared memory as [row][128 features]; then a warp takes every fourth row with four consecutive
    // features per lane, so that stores are whole lines and the row maximum of the LM head is one reduction over the warp.
    pdl_wait();   // outputs of this kernel may still be read by the previous one's consumers
    const int q = warp & 3;                       // TMEM lane quarter this warp may read
    const int grp = (warp - 2) >> 2, w4 = (warp - 2) & 3;
    const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16);
    const uint32_t stg = smem_u32(staging) + grp * 2 * kPassBytes;
    const uint32_t acc_empty0 = cluster_addr(smem_u32(&ctl->acc_empty[0]), 0);
    auto group_sync = [&] { asm volatile("bar.sync %0, 128;" ::"r"(1 + grp) : "memory"); };
    auto all_sync = [&] { asm volatile("bar.sync 3, 256;" ::: "memory"); };
    uint32_t buf = 0;
    PairItem t;
    for (int j = 0; pair_item(g, pair, P, j, t); ++j) {
      const int b = j & 1;
      if constexpr (EPI == EPI_SWIGLU) {
        const int r = (int)threadIdx.x - 64;
        if (g.ss && r < t.rows && t.m0 + r < g.M) {
          const float *p = g.ss + (size_t)(t.m0 + r) * g.ss_tiles;
          float f = 0.f;
#pragma unroll 8
          for (int i = 0; i < g.ss_tiles; ++i) f += p[i];
          ctl->rs[b][r] = rsqrtf(f * g.inv_d + g.eps);
        }
      }
      bool ok = __all_sync(0xffffffffu, mbar_wait_cluster(smem_u32(&ctl->acc_full[b]), (j >> 1) & 1));
      if (!ok && lane == 0) atomicExch(g.err, DEV_TIMEOUT_TMEM);
      tc_fence_after();
      ok = ok && (*reinterpret_cast<volatile uint32_t *>(&ctl->abort_flag) == 0);
      // (the epilogue warps leave together: whoever is left behind would wait in a barrier for good)
      uint32_t all_ok;
      asm volatile(
          "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.and.pred q, 3, 256, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
          : "=r"(all_ok)
          : "r"((uint32_t)ok)
          : "memory");
      if (!all_ok) break;
      const int blk = 2 * t.wt + rank, n = blk * kBoxN + lane * 4;   // this lane's features n .. n + 3 in the second pass
      const int rows = blk < n_blocks ? min(t.rows, g.M - t.m0) : 0;
      const uint32_t tacc = taddr + b * set_cols;
      // what becomes of row r of the chunk, by a whole warp
      auto finish = [&](int r, float4 v) {
        const int m = t.m0 + r;
        if constexpr (EPI == EPI_SWIGLU) {
          if (g.ss) {
            const float f = ctl->rs[b][r];
            v.x *= f; v.y *= f; v.z *= f; v.w *= f;
          }
        }
        if constexpr (EPI == EPI_PARTIAL) {
          *reinterpret_cast<float4 *>(g.out + ((size_t)t.slice * g.out_rows + m) * g.N + n) = v;
        } else if constexpr (EPI == EPI_LOGITS) {
          *reinterpret_cast<float4 *>(g.out + (size_t)m * g.N + n) = v;
          // order-preserving map of the float to an unsigned word; ties resolve to the lowest id (lowest lane, then
          // lowest of its four)
          const float f[4] = {v.x, v.y, v.z, v.w};
          uint32_t best = 0;
          int bi = 0;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            uint32_t u = __float_as_uint(f[i]);
            u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
            if (u > best) { best = u; bi = i; }
          }
          const uint32_t top = __reduce_max_sync(0xffffffffu, best);
          if (lane == __ffs(__ballot_sync(0xffffffffu, best == top)) - 1)
            atomicMax(g.amax + (size_t)m * kAmaxStride, ((unsigned long long)top << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)(n + bi)));
        } else {  // EPI_SWIGLU: even feature row = gate_f, odd = up_f, f = n / 2
          __nv_bfloat16 h0, l0, h1, l1;
          split_bf16(v.x / (1.f + __expf(-v.x)) * v.y, h0, l0);
          split_bf16(v.z / (1.f + __expf(-v.z)) * v.w, h1, l1);
          const int F = g.N >> 1, f = n >> 1;
          *reinterpret_cast<__nv_bfloat162 *>(g.act_out + (size_t)m * F + f) = __halves2bfloat162(h0, h1);
          if (g.out_planes == 2)
            *reinterpret_cast<__nv_bfloat162 *>(g.act_out + ((size_t)g.act_rows + m) * F + f) = __halves2bfloat162(l0, l1);
        }
      };
      // slab (cut tile, slice, CTA of the pair): [chunk rows][128 features]
      const bool slab = EPI != EPI_PARTIAL && t.cut >= 0;
      auto slab_at = [&](int slice) { return g.slab + ((size_t)(t.cut * g.pieces + slice) * 2 + rank) * g.chunk_rows * kBoxN + lane * 4; };
      float *own = slab ? slab_at(t.slice) : nullptr;
      for (int c0 = grp * kPassRows; c0 < t.rows; c0 += 2 * kPassRows, buf ^= 1) {
        uint32_t r[16];
        if (apart) {
          // rows of either half: value plane, then remainder plane (halves come in eights)
          uint32_t a[8], b8[8], c[8], e[8];
          const int h = t.rows >> 1, c1 = c0 + 8, k0 = c0 < h ? c0 : c0 + h, k1 = c1 < h ? c1 : c1 + h;
          tmem_ld8(tacc + k0, a);
          tmem_ld8(tacc + k0 + h, b8);
          tmem_ld8(tacc + k1, c);
          tmem_ld8(tacc + k1 + h, e);
          tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            r[i] = __float_as_uint(__uint_as_float(a[i]) + __uint_as_float(b8[i]));
            r[8 + i] = __float_as_uint(__uint_as_float(c[i]) + __uint_as_float(e[i]));
          }
        } else {
          tmem_ld16(tacc + c0, r);
          tmem_wait_ld();
        }
        const uint32_t at = stg + buf * kPassBytes;   // (two buffers in turn: a barrier per pass)
#pragma unroll
        for (int i = 0; i < 16; ++i) st_shared_f32(at + (i * kBoxN + q * 32 + lane) * 4, __uint_as_float(r[i]));
        if (c0 + 2 * kPassRows >= t.rows) {   // (the sums are out of tensor memory when a warp has read its last columns)
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(acc_empty0 + b * 8);
        }
        group_sync();
#pragma unroll
        for (int i = 0; i < kPassRows / 4; ++i) {
          const int rr = w4 + 4 * i;
          const uint4 raw = ld_shared_v4(at + (rr * kBoxN + lane * 4) * 4);
          if (c0 + rr >= rows) continue;
          const float4 v = make_float4(__uint_as_float(raw.x), __uint_as_float(raw.y), __uint_as_float(raw.z), __uint_as_float(raw.w));
          if (slab) *reinterpret_cast<float4 *>(own + (size_t)(c0 + rr) * kBoxN) = v;
          else finish(c0 + rr, v);
        }
      }
      if (grp * kPassRows >= t.rows) {   // (a chunk of one pass: the second group has no columns)
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(acc_empty0 + b * 8);
      }
      if (slab) {
        // the last CTA to write a slab of this tile adds them all, in K order
        __threadfence();
        all_sync();
        if (threadIdx.x == 64) {
          unsigned int *n_done = g.n_done + 2 * t.cut + rank;
          const bool last = atomicAdd(n_done, 1u) == (unsigned)g.pieces - 1;
          if (last) *n_done = 0;   // (for the next launch)
          __threadfence();
          ctl->last = last;
        }
        all_sync();
        if (ctl->last) {
          // (four rows of a warp and up to kFoldAhead slabs are on their way at a time: a row and a slab after the other took
          // 25 us for 256 rows of two slabs)
          for (int r0 = warp - 2; r0 < rows; r0 += 32) {
            float4 v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int s0 = 0; s0 < g.pieces; s0 += kFoldAhead) {
              float4 p[kFoldAhead][4];
#pragma unroll
              for (int s = 0; s < kFoldAhead; ++s)
#pragma unroll
                for (int i = 0; i < 4; ++i)
                  p[s][i] = ld_global_v4_if(slab_at(s0 + s) + (size_t)(r0 + 8 * i) * kBoxN, s0 + s < g.pieces && r0 + 8 * i < rows);
#pragma unroll
              for (int s = 0; s < kFoldAhead; ++s)
#pragma unroll
                for (int i = 0; i < 4; ++i)
                  if (s0 + s < g.pieces) { v[i].x += p[s][i].x; v[i].y += p[s][i].y; v[i].z += p[s][i].z; v[i].w += p[s][i].w; }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              if (r0 + 8 * i >= rows) break;
              finish(r0 + 8 * i, v[i]);
            }
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncwarp();
  cluster_arrive();   // (the other CTA's products read this one's shared memory, and its commits and arrivals end here)
  cluster_wait();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, alloc_cols);
  }
  if (threadIdx.x == 0 && g.stamp) stamp_max(g.stamp + 3);
}

static size_t pair_smem_bytes(int stages, int planes, int rows) {
  return (size_t)stages * (kBoxBytes + planes * rows / 2 * kBlockK * 2) + kStagingBytes + sizeof(PairSmemCtl) + 1024;
}

template <int EPI>
static cudaError_t launch_pair_one(const CUtensorMap &tw, const CUtensorMap &ta, const CUtensorMap &ta_less, const PairArgs &g,
                                   dim3 grid, size_t smem, cudaStream_t st, bool pdl) {
  static PerDeviceOnce once;
  int dev_ = -1;
  if (once.needed(&dev_)) {
    cudaError_t e = cudaFuncSetAttribute(gemm_pair_kernel<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
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
  return cudaLaunchKernelEx(&cfg, gemm_pair_kernel<EPI>, tw, ta, ta_less, g);
}

// How a launch is cut up.  Rows: as few chunks as hold them (below 144 rows a k-block is bound by its bytes from L2, so more and
// smaller chunks only cost), alike to within one step of the instruction's N.
PairPlan plan_gemm_pair(int N, int M, int n_kblocks, int planes, bool fold, int pairs, int max_pieces, size_t slab_room) {
  PairPlan p{};
  const int steps = (M + 15) / 16;
  p.chunks = (M + 255) / 256;
  p.rows = (steps + p.chunks - 1) / p.chunks * 16;
  p.n_wide = steps - p.chunks * (p.rows / 16 - 1);
  p.tiles = p.whole = (N + 255) / 256 * p.chunks;
  p.pieces = 1;
  // a k-block: its products, its bytes from L2 (16 KB and 128 a row for each CTA), or the weights from HBM
  const double r256 = p.rows / 256.0;
  const double kb = std::max(std::max(0.05 + 0.32 * planes * r256, 0.17 + 0.17 * planes * r256), 0.37 / p.chunks);
  p.us = 1e30;
  if (!fold) {
    // every slice adds a slab that this kernel writes and the next one reads
    for (int s = 1; s <= max_pieces && (s == 1 || s <= n_kblocks / 4); ++s) {
      const double t = (p.tiles * s + pairs - 1) / pairs * (kb * n_kblocks / s + 1.0) + 6.3 + rows_slab_us(M, N) * s;
      if (t < p.us - 1e-9) { p.us = t; p.pieces = s; }
    }
    if (p.pieces > 1) p.whole = 0;
  } else {
    const int q = p.tiles / pairs, r = p.tiles % pairs;
    const double out = 3.0 + 8.0 * r256;   // the last tile's way out
    const double uncut = r ? kb * n_kblocks + 1.0 : 0.0;
    double best = uncut;                             // of what comes on top of q whole tiles each
    for (int s = 2; r && s <= max_pieces && s <= n_kblocks / 4; ++s) {
      if ((size_t)r * s * 2 * p.rows * kBoxN > slab_room) break;
      // (a piece costs at least its sums' way out; what the adding takes beyond a whole tile's products shows as well)
      const int mine = (r * s + pairs - 1) / pairs;
      const double add = 10.0 * r256 * ((s + kFoldAhead - 1) / kFoldAhead) + 5.0 * r256 * mine;
      const double t = mine * std::max(kb * n_kblocks / s + 2.0, 6.0 * r256) + std::max(0.0, add - (q ? kb * n_kblocks : 0.0));
      // (slabs are traffic that the count above takes for hidden: not for a few per cent -- LM head of the 1B shape at 112 rows, 57
      // tiles left for 74 pairs, 99 us uncut against 112)
      if (t < best - 1e-9 && t < 0.75 * uncut) { best = t; p.pieces = s; }
    }
    if (p.pieces > 1) p.whole = q * pairs;
    // (tiles of few k-blocks: an epilogue takes as long as the next tile's products, and memory from them; 1B shape, gate-up of 768
    // rows 91 us against the row-major kernel's 89, of 475 54 against 61)
    const double between = planes == 2 && n_kblocks < 48 ? 2.5 * r256 * r256 * std::max(0, q - (r ? 0 : 1)) : 0.0;
    p.us = q * (kb * n_kblocks + 0.5) + between + best + out;
  }
  p.pairs = std::min(pairs, p.whole + (p.tiles - p.whole) * p.pieces);
  return p;
}

// `ta`, `ta_less`: activation maps whose boxes hold half of plan.rows and half of plan.rows - 16 rows (the second is not used
// where plan.n_wide == plan.chunks).  N must be a multiple of 128.
cudaError_t launch_gemm_pair(int epi, const CUtensorMap &tw, const CUtensorMap &ta, const CUtensorMap &ta_less, PairArgs g,
                             const PairPlan &plan, size_t smem_limit, cudaStream_t st, bool pdl) {
  if (g.ss && plan.rows > 128) return cudaErrorInvalidValue;
  if (plan.pieces < 1 || plan.pieces > g.n_kblocks || g.N % kBoxN || plan.rows % 16 || plan.rows < 16 || plan.rows > 256 || plan.pairs < 1)
    return cudaErrorInvalidValue;
  g.chunk_rows = plan.rows;
  g.n_wide = plan.n_wide;
  g.chunks = plan.chunks;
  g.n_tiles = plan.tiles;
  g.n_whole = plan.whole;
  g.pieces = plan.pieces;
  g.stages = kMaxStages;
  while (g.stages > 2 && pair_smem_bytes(g.stages, g.planes, plan.rows) > smem_limit) --g.stages;
  const size_t smem = pair_smem_bytes(g.stages, g.planes, plan.rows);
  if (smem > smem_limit) return cudaErrorInvalidConfiguration;
  const dim3 grid(2 * plan.pairs);
  switch (epi) {
    case EPI_PARTIAL: return launch_pair_one<EPI_PARTIAL>(tw, ta, ta_less, g, grid, smem, st, pdl);
    case EPI_SWIGLU: return launch_pair_one<EPI_SWIGLU>(tw, ta, ta_less, g, grid, smem, st, pdl);
    case EPI_LOGITS: return launch_pair_one<EPI_LOGITS>(tw, ta, ta_less, g, grid, smem, st, pdl);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace ts
