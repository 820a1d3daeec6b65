// Weight-streaming GEMM for the verify step's dense projections (QKV, O, gate-up, down, LM head):
//     out[m][n] = sum_k act[m][k] * W[n][k]
// with few rows m (the verified positions) and a large weight matrix read exactly once.
//
// The weight matrix is stored as contiguous 128 x 64 blocks (one TMA box each).
// Operands are swapped with respect to the usual layout so that the 128-row dimension of the
// tensor-core instruction runs over output features: a CTA owns 128 rows of W (operand A, K-major,
// 16 KB per 64-wide k-block) and the step's activation rows, at most 80 or, with one plane, 96 (operand B).  Activations can
// be fed as a (hi, lo) bf16 pair stacked along the instruction's N dimension, so one MMA multiplies
// the weight tile with both halves; the epilogue adds the two column groups.  The accumulator lives
// in tensor memory: lane = output feature, column = activation row.
//
// Roles: warp 0 = TMA producer, warp 1 = TMEM allocation + MMA issue, warps 2..5 = epilogue.
// Every wait is bounded; on expiry the CTA records an error word and leaves through the normal exit.
#include <cuda_fp16.h>

#include "kernels.h"

namespace ts {

static constexpr int kBlockK = 64;                 // k-block: 64 bf16 = 128 bytes per row
static constexpr int kTileN = 128;                 // weight rows per CTA
static constexpr int kWBytes = kTileN * kBlockK * 2;
static constexpr int kMaxStages = 8;
static constexpr int kPushRows = 16;               // most rows whose sums are sent (see launch_gemm)

struct __align__(16) GemmSmemCtl {
  uint64_t full[kMaxStages];
  uint64_t empty[kMaxStages];
  uint64_t tmem_full;
  uint64_t got;            // clusters that send their sums: those of this CTA's rows are here, from all K slices
  uint32_t tmem_base;
  uint32_t abort_flag;
  float rs[128];  // per activation row: 1 / rms of the input (1 where the input is normalised already)
};

__device__ __forceinline__ __half to_half_sat(float x) { return __float2half_rn(fminf(fmaxf(x, -65504.f), 65504.f)); }
__device__ __forceinline__ __half2 to_half2_sat(float a, float b) { return __halves2half2(to_half_sat(a), to_half_sat(b)); }
// rounding remainder of a value stored as fp16 (dropped where the value saturates)
__device__ __forceinline__ float half_rest(float x, __half h) { return fabsf(x) <= 65504.f ? x - __half2float(h) : 0.f; }

__device__ __forceinline__ void epilogue_sync() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

// where row m's K/V of `head` (counted over Q, K and V heads) go, in rows of hd elements of the layer's K or V pages
__device__ __forceinline__ long long kv_place(const GemmArgs &g, int m, int head) {
  const int kh = head < g.Hq + g.Hkv ? head - g.Hq : head - g.Hq - g.Hkv, slot = g.in.slot[m];
  const int page = g.in.block_tab[(size_t)g.in.row_seq[m] * g.in.pages_per_seq + (slot >> 4)];
  return ts_in_range(g.in.ck, CHK_PAGE_APPEND, page, g.in.ck.max_pages) ? ((long long)page * g.Hkv + kh) * 16 + (slot & 15) : -1;
}
__device__ __forceinline__ void add4(float4 &s, const float4 &v) { s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w; }

// PUSH (QKV, RESID): sums are sent to the CTAs that finish the rows, see launch_gemm.  (A template argument: a branch at each load
// of a sum keeps the loads from being issued together, 0.7 to 1.2 us per launch.)
template <int EPI, bool PUSH>
__global__ void __launch_bounds__(192, 1)
gemm_ws_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_a,
               const GemmArgs g) {
  // 1024-byte alignment is required by the 128-byte swizzle pattern: the declared one holds (no room is spent on rounding up)
  extern __shared__ __align__(1024) uint8_t smem[];
#ifdef TS_DEBUG_BOUNDS
  if (threadIdx.x == 0 && (smem_u32(smem) & 1023u)) atomicCAS(g.err, 0, DEV_BOUNDS + CHK_SMEM);
#endif
  const int a_bytes = g.planes * g.Mc * kBlockK * 2;
  const int stage_bytes = kWBytes + a_bytes;
  GemmSmemCtl *ctl = reinterpret_cast<GemmSmemCtl *>(smem + (size_t)g.stages * stage_bytes);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n0 = blockIdx.x * kTileN;
  constexpr bool kCluster = EPI == EPI_QKV || EPI == EPI_RESID;
  const int split = blockIdx.y;   // (with kCluster: the CTA's rank in its cluster, which spans the K slices of one tile)
  // balanced cut of the k-blocks into gridDim.y runs
  const int kb0 = (int)(((long long)split * g.n_kblocks) / (int)gridDim.y);
  const int kb1 = (int)(((long long)(split + 1) * g.n_kblocks) / (int)gridDim.y);
  const int nkb = kb1 - kb0;
  const uint32_t ncols = g.planes * g.Mc;
  uint32_t alloc_cols = 32;
  while (alloc_cols < ncols) alloc_cols <<= 1;

  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&tmap_w);
    tma_prefetch_desc(&tmap_a);
    for (int s = 0; s < g.stages; ++s) {
      mbar_init(smem_u32(&ctl->full[s]), 1);
      mbar_init(smem_u32(&ctl->empty[s]), 1);
    }
    mbar_init(smem_u32(&ctl->tmem_full), 1);
    ctl->abort_flag = 0;
    if constexpr (kCluster) mbar_init(smem_u32(&ctl->got), 1);
    fence_barrier_init();
    if constexpr (kCluster) {
      const int C = (int)gridDim.y, per = (g.M + C - 1) / C;
      if constexpr (PUSH) mbar_expect_tx(smem_u32(&ctl->got), C * min(per, max(0, g.M - split * per)) * kTileN * 4);
    }
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&ctl->tmem_base), alloc_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if constexpr (PUSH) cluster_arrive();   // (this CTA's barrier is set up: waited for before the first sums are sent)
  const uint32_t tmem_base = ctl->tmem_base;
  if (threadIdx.x == 0) stamp_min(g.stamp);
  // Let the next kernel launch now: it waits (griddepcontrol.wait) for this one to finish before it touches
  // dependent data, so only its launch latency and its own prologue (weight prefetch) move forward.  Placed after
  // this CTA holds its resources, so a waiting dependent can never starve an earlier kernel.
  pdl_launch_dependents();

  if (warp == 0) {
    // ------------------------------------------------------------------ producer
    if (lane == 0 && nkb > 0) {
      const uint64_t pol_w = policy_evict_first(), pol_a = policy_evict_last();
      const int pre = min(g.stages, nkb);
      // weights do not depend on the previous kernel: start streaming them before the
      // programmatic-dependency wait, activations after it
      for (int it = 0; it < pre; ++it) {
        uint32_t bar = smem_u32(&ctl->full[it]);
        mbar_expect_tx(bar, stage_bytes);
        tma_load_2d(smem_u32(smem + (size_t)it * stage_bytes), &tmap_w, 0, w_block(blockIdx.x, kb0 + it, g.N / kTileN, g.n_kblocks) * kTileN, bar, pol_w);
      }
      pdl_wait();
      stamp_waited(g.stamp);
      for (int it = 0; it < pre; ++it) {
        uint32_t bar = smem_u32(&ctl->full[it]);
        tma_load_3d(smem_u32(smem + (size_t)it * stage_bytes + kWBytes), &tmap_a, (kb0 + it) * kBlockK, 0, 0,
                    bar, pol_a);
      }
      // slot and round parity are carried along: an integer division per k-block would be a large part of
      // this single thread's time budget per block
      int s = (pre == g.stages) ? 0 : pre;
      uint32_t ph = (pre == g.stages) ? 1 : 0;
      for (int it = pre; it < nkb; ++it) {
        if (!mbar_wait(smem_u32(&ctl->empty[s]), ph ^ 1)) {
          atomicExch(g.err, DEV_TIMEOUT_EMPTY);
          break;
        }
        uint32_t bar = smem_u32(&ctl->full[s]);
        mbar_expect_tx(bar, stage_bytes);
        uint32_t dst = smem_u32(smem + (size_t)s * stage_bytes);
        tma_load_2d(dst, &tmap_w, 0, w_block(blockIdx.x, kb0 + it, g.N / kTileN, g.n_kblocks) * kTileN, bar, pol_w);
        tma_load_3d(dst + kWBytes, &tmap_a, (kb0 + it) * kBlockK, 0, 0, bar, pol_a);
        if (++s == g.stages) { s = 0; ph ^= 1; }
      }
    } else if (lane == 0) {
      pdl_wait();
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issue
    // The whole warp walks the loop and the waits; one elected lane issues the instructions of a k-block and its
    // commit (a lone lane in a divergent branch needs about 50 cycles per tensor-core instruction, this form 22).
    {
      const uint32_t idesc = umma_idesc_bf16(kTileN, ncols);
      bool ok = true;
      int s = 0;
      uint32_t ph = 0;
      for (int it = 0; it < nkb; ++it) {
        if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&ctl->full[s]), ph))) {   // (all lanes leave together)
          if (lane == 0) atomicExch(g.err, DEV_TIMEOUT_FULL);
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t sa = smem_u32(smem + (size_t)s * stage_bytes);
        const uint64_t da = umma_desc_sw128(sa), db = umma_desc_sw128(sa + kWBytes);
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < kBlockK / 16; ++kk) {
            // 16 bf16 along K = 32 bytes = 2 descriptor address units
            umma_bf16(tmem_base, da + 2 * kk, db + 2 * kk, idesc, (it | kk) != 0);
          }
          umma_commit(smem_u32(&ctl->empty[s]));
        }
        __syncwarp();
        if (++s == g.stages) { s = 0; ph ^= 1; }
      }
      if (elect_one()) {
        if (!ok) ctl->abort_flag = 1;
        umma_commit(smem_u32(&ctl->tmem_full));
      }
      __syncwarp();
    }
  } else {
    // ------------------------------------------------------------------ epilogue (warps 2..5)
    // Two passes through the ring's shared memory (free by now: every load was consumed by a product that has
    // completed).  First thread <-> feature: the accumulator's columns, both planes added, go to [row][128 features].
    // Then a warp takes every fourth row with four consecutive features per lane, so that global stores are whole lines
    // and the row maximum of the LM head is one reduction over the warp per row.  (With a thread keeping its one feature
    // a row's argmax took ten shuffles per warp and row and its SwiGLU stores were 32-byte pieces: the LM head of the 8B
    // shape took 286 us at 32 rows and 180 at one, same weights.)
    // With the K slices of a tile in one cluster (QKV, O, down) the rows are dealt out between the two passes: CTA r of C
    // finishes rows [r, r + 1) * ceil(M / C), adding the C slices' sums in slice order out of the other CTAs' shared memory
    // -- the same order whatever the number of rows.  Before, the slices went to L2 as slabs that a norm or rotary kernel
    // of its own folded: three launches and their boundaries more per layer (8B shape at 32 rows: QKV + rotary 12.8 -> 11.6
    // us, O + norm 10.9 -> 9.8, down + norm 20.6 -> 19.0; 1B shape at 8 rows 38 -> 34 us per layer).  Of a launch's time the
    // exchange costs about 2 us: 0.6 for the slowest CTA of the cluster, 0.4 - 1.0 for the reads, the rest stores.
    pdl_wait();   // outputs of this kernel may still be read by the previous one's consumers
    if constexpr (EPI == EPI_QKV || EPI == EPI_SWIGLU) {
      const int m = (int)threadIdx.x - 64;
      if (m < g.M) {
        float s = 0.f;
        if (g.ss) {
          const float *p = g.ss + (size_t)m * g.ss_tiles;
#pragma unroll 8
          for (int i = 0; i < g.ss_tiles; ++i) s += p[i];
          s = rsqrtf(s * g.inv_d + g.eps);
        } else {
          s = 1.f;
        }
        ctl->rs[m] = s;
      }
    }
    const int C = kCluster ? (int)gridDim.y : 1;
    const int rows_per = (g.M + C - 1) / C, m_beg = kCluster ? split * rows_per : 0, m_end = min(g.M, m_beg + rows_per);
    const int n = n0 + lane * 4;                  // this lane's features n .. n + 3 in the second pass
    // what the second pass needs besides the sums is on its way before the sums are complete
    constexpr int kPre = 2;
    float4 pre[kPre], gn = make_float4(0.f, 0.f, 0.f, 0.f);
    int head = 0, ei = 0, half = 0;
    long long kv_row[kPre];                       // K/V heads: the row's place in the pages (in rows of hd elements), -1: none
    if constexpr (EPI == EPI_RESID) {
      gn = *reinterpret_cast<const float4 *>(g.gain + n);
#pragma unroll
      for (int i = 0; i < kPre; ++i) {
        const int m = m_beg + (warp - 2) + 4 * i;
        if (m < m_end) pre[i] = *reinterpret_cast<const float4 *>(g.x + (size_t)m * g.N + n);
      }
    } else if constexpr (EPI == EPI_QKV) {
      // QKV weight rows are stored with rotary partners adjacent: feature 2e of a head = element e, 2e + 1 = element
      // e + hd/2; this lane has the pairs ei and ei + 1 of one head
      head = n / g.hd;
      half = g.hd >> 1;
      ei = (n - head * g.hd) >> 1;
      if (head < g.Hq + g.Hkv) {
#pragma unroll
        for (int i = 0; i < kPre; ++i) {
          const int m = m_beg + (warp - 2) + 4 * i;
          if (m < m_end) {
            const int pos = g.in.pos[m];
            pre[i] = ts_in_range(g.in.ck, CHK_POSITION, pos, g.in.ck.max_ctx)
                         ? *reinterpret_cast<const float4 *>(g.rope_tab + (size_t)pos * half + ei)
                         : make_float4(1.f, 0.f, 1.f, 0.f);
          }
        }
      }
      if (head >= g.Hq) {
#pragma unroll
        for (int i = 0; i < kPre; ++i) {
          const int m = m_beg + (warp - 2) + 4 * i;
          kv_row[i] = m < m_end ? kv_place(g, m, head) : -1;
        }
      }
    }
    bool ok = true;
    if (nkb > 0) {
      ok = mbar_wait(smem_u32(&ctl->tmem_full), 0);
      if (!ok && lane == 0) atomicExch(g.err, DEV_TIMEOUT_TMEM);
      ok = __all_sync(0xffffffffu, ok);
    }
    tc_fence_after();
    ok = ok && (*reinterpret_cast<volatile uint32_t *>(&ctl->abort_flag) == 0);
    const int q = warp & 3;                       // TMEM lane quarter this warp may read
    const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16);
    const uint32_t stg = smem_u32(smem);
    // Sums sent (see launch_gemm): [slice][row of the CTA's][128 features] behind the control block of the CTA that finishes the rows.
    const uint32_t inbox = smem_u32(ctl + 1), got = smem_u32(&ctl->got);
    int to_row = 0, to = 0;    // the next row is row `to_row` of CTA `to`
    uint32_t to_box = 0, to_bar = 0;
    auto send_to = [&](int r) {
      to = r;
      to_row = 0;
      to_box = cluster_addr(inbox + (split * rows_per * kTileN + q * 32 + lane) * 4, r);
      to_bar = cluster_addr(got, r);
    };
    if constexpr (PUSH) {
      cluster_wait();   // (all CTAs of the cluster are set up: long since)
      send_to(0);
    }
    // (columns past the step's last row are read too and never used)
    auto put = [&](int c, uint32_t lo, uint32_t hi) {
      const float v = __uint_as_float(lo) + (g.planes == 2 ? __uint_as_float(hi) : 0.f);
      if constexpr (!PUSH) {
        st_shared_f32(stg + (c * kTileN + q * 32 + lane) * 4, v);
      } else if (c < g.M && ok) {
        st_async_f32(to_box + to_row * kTileN * 4, v, to_bar);
        if (++to_row == rows_per && c + 1 < g.M) send_to(to + 1);
      }
    };
    int c0 = 0;
    for (; c0 + 16 <= g.Mc; c0 += 16) {
      uint32_t r[16], r2[16];
      tmem_ld16(taddr + c0, r);
      if (g.planes == 2) tmem_ld16(taddr + g.Mc + c0, r2);
      tmem_wait_ld();
#pragma unroll
      for (int j = 0; j < 16; ++j) put(c0 + j, r[j], r2[j]);
    }
    if (c0 < g.Mc) {
      uint32_t r[8], r2[8];
      tmem_ld8(taddr + c0, r);
      if (g.planes == 2) tmem_ld8(taddr + g.Mc + c0, r2);
      tmem_wait_ld();
#pragma unroll
      for (int j = 0; j < 8; ++j) put(c0 + j, r[j], r2[j]);
    }
    if constexpr (PUSH) {
      if (m_beg < m_end) {
        const bool here = __all_sync(0xffffffffu, mbar_wait_cluster(got, 0));
        if (!here) {
          if (lane == 0) atomicExch(g.err, DEV_TIMEOUT_TMEM);
          *reinterpret_cast<volatile uint32_t *>(&ctl->abort_flag) = 1;
        }
        ok = ok && here;
      }
    } else if constexpr (kCluster) {
      __syncwarp();
      cluster_arrive();
      cluster_wait();
    } else {
      epilogue_sync();
    }
    // (a warp's rows two at a time: all their partial sums are fetched before the first is worked on)
    bool left = !kCluster || PUSH;   // this CTA has read all that it needs from the others
#pragma unroll 1
    for (int mg = m_beg + warp - 2, i0 = 0; ok && mg < m_end; mg += 8, i0 += 2) {
      float4 sum[2];
      if constexpr (kCluster) {
        float4 p[2][8];
        const bool two = mg + 4 < m_end;
        auto part = [&](int m, int c) {
          if constexpr (PUSH) {
            const uint4 v = ld_shared_v4(inbox + ((c * rows_per + m - m_beg) * kTileN + lane * 4) * 4);
            return make_float4(__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w));
          } else {
            return ld_cluster_v4(stg + (m * kTileN + lane * 4) * 4, c);
          }
        };
#pragma unroll
        for (int c = 0; c < 8; ++c)
          if (c < C) p[0][c] = part(mg, c);
        if (two) {
#pragma unroll
          for (int c = 0; c < 8; ++c)
            if (c < C) p[1][c] = part(mg + 4, c);
        }
        sum[0] = p[0][0];
#pragma unroll
        for (int c = 1; c < 8; ++c)
          if (c < C) add4(sum[0], p[0][c]);
        if (two) {
          sum[1] = p[1][0];
#pragma unroll
          for (int c = 1; c < 8; ++c)
            if (c < C) add4(sum[1], p[1][c]);
        }
        if (!PUSH && mg + 8 >= m_end) {   // (nothing is left to read: the others may go; they are waited for at the end)
          __syncwarp();
          cluster_arrive();
          left = true;
        }
      }
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int m = mg + 4 * i;
        if (m >= m_end) break;
        float v[4];
        if constexpr (kCluster) {
          v[0] = sum[i].x; v[1] = sum[i].y; v[2] = sum[i].z; v[3] = sum[i].w;
        } else {
          const uint4 raw = ld_shared_v4(stg + (m * kTileN + lane * 4) * 4);
          v[0] = __uint_as_float(raw.x); v[1] = __uint_as_float(raw.y); v[2] = __uint_as_float(raw.z); v[3] = __uint_as_float(raw.w);
        }
        if constexpr (EPI == EPI_QKV || EPI == EPI_SWIGLU) {
          const float s = ctl->rs[m];
#pragma unroll
          for (int j = 0; j < 4; ++j) v[j] *= s;
        }
        if constexpr (EPI == EPI_RESID) {
          float4 xv = i0 == 0 ? pre[i] : *reinterpret_cast<const float4 *>(g.x + (size_t)m * g.N + n);
          xv.x += v[0]; xv.y += v[1]; xv.z += v[2]; xv.w += v[3];
          *reinterpret_cast<float4 *>(g.x + (size_t)m * g.N + n) = xv;
          const float sq = warp_sum(xv.x * xv.x + xv.y * xv.y + xv.z * xv.z + xv.w * xv.w);
          if (lane == 0) g.ss_out[(size_t)m * gridDim.x + blockIdx.x] = sq;
          if (g.h_out) {
            __align__(8) __nv_bfloat16 hi[4], lo[4];
            split_bf16(xv.x * gn.x, hi[0], lo[0]);
            split_bf16(xv.y * gn.y, hi[1], lo[1]);
            split_bf16(xv.z * gn.z, hi[2], lo[2]);
            split_bf16(xv.w * gn.w, hi[3], lo[3]);
            *reinterpret_cast<uint2 *>(g.h_out + (size_t)m * g.N + n) = *reinterpret_cast<const uint2 *>(hi);
            if (g.out_planes == 2)
              *reinterpret_cast<uint2 *>(g.h_out + ((size_t)g.act_rows + m) * g.N + n) = *reinterpret_cast<const uint2 *>(lo);
          }
        } else if constexpr (EPI == EPI_QKV) {
          float a0 = v[0], b0 = v[1], a1 = v[2], b1 = v[3];   // elements ei, ei + hd/2, ei + 1, ei + 1 + hd/2
          if (head < g.Hq + g.Hkv) {
            float4 cs;
            if (i0 == 0) {
              cs = pre[i];
            } else {
              const int pos = g.in.pos[m];
              cs = ts_in_range(g.in.ck, CHK_POSITION, pos, g.in.ck.max_ctx)
                       ? *reinterpret_cast<const float4 *>(g.rope_tab + (size_t)pos * half + ei)
                       : make_float4(1.f, 0.f, 1.f, 0.f);
            }
            const float ra0 = a0 * cs.x - b0 * cs.y, rb0 = b0 * cs.x + a0 * cs.y;
            const float ra1 = a1 * cs.z - b1 * cs.w, rb1 = b1 * cs.z + a1 * cs.w;
            a0 = ra0; b0 = rb0; a1 = ra1; b1 = rb1;
          }
          const __half2 ha = to_half2_sat(a0, a1), hb = to_half2_sat(b0, b1);
          if (head < g.Hq) {
            // the query as an fp16 pair (value, rounding remainder): the score product adds both, so the 11 bits of
            // fp16 do not limit the scores
            const size_t qo = ((size_t)m * g.Hq + head) * g.hd + ei;
            *reinterpret_cast<__half2 *>(g.q_out + qo) = ha;
            *reinterpret_cast<__half2 *>(g.q_out + qo + half) = hb;
            *reinterpret_cast<__half2 *>(g.q_lo_out + qo) = __floats2half2_rn(half_rest(a0, __low2half(ha)), half_rest(a1, __high2half(ha)));
            *reinterpret_cast<__half2 *>(g.q_lo_out + qo + half) = __floats2half2_rn(half_rest(b0, __low2half(hb)), half_rest(b1, __high2half(hb)));
          } else {
            const long long at = i0 == 0 ? kv_row[i] : kv_place(g, m, head);
            if (at >= 0) {
              __half *dst = (head < g.Hq + g.Hkv ? g.k_pages : g.v_pages) + at * g.hd + ei;
              *reinterpret_cast<__half2 *>(dst) = ha;
              *reinterpret_cast<__half2 *>(dst + half) = hb;
            }
          }
        } else if constexpr (EPI == EPI_LOGITS) {
          *reinterpret_cast<float4 *>(g.out + (size_t)m * g.N + n) = make_float4(v[0], v[1], v[2], v[3]);
          // order-preserving map of the float to an unsigned word; ties resolve to the lowest id (lowest lane, then
          // lowest of its four)
          uint32_t best = 0;
          int bi = 0;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            uint32_t u = __float_as_uint(v[j]);
            u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
            if (u > best) { best = u; bi = j; }
          }
          const uint32_t top = __reduce_max_sync(0xffffffffu, best);
          if (lane == __ffs(__ballot_sync(0xffffffffu, best == top)) - 1)
            atomicMax(g.amax + (size_t)m * kAmaxStride, ((unsigned long long)top << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)(n + bi)));
        } else {  // EPI_SWIGLU: even feature row = gate_f, odd = up_f, f = n / 2
          __nv_bfloat16 h0, l0, h1, l1;
          split_bf16(v[0] / (1.f + __expf(-v[0])) * v[1], h0, l0);
          split_bf16(v[2] / (1.f + __expf(-v[2])) * v[3], h1, l1);
          const int F = g.N >> 1, f = n >> 1;
          *reinterpret_cast<__nv_bfloat162 *>(g.act_out + (size_t)m * F + f) = __halves2bfloat162(h0, h1);
          if (g.out_planes == 2)
            *reinterpret_cast<__nv_bfloat162 *>(g.act_out + ((size_t)g.act_rows + m) * F + f) = __halves2bfloat162(l0, l1);
        }
      }
    }
    if constexpr (kCluster) {
      if (!left) {
        __syncwarp();
        cluster_arrive();
      }
    }
  }
  if constexpr (kCluster) {
    // (every thread of the cluster takes part in both barriers: the sums are in shared memory, then: nobody reads mine
    // any more; the waits inside the roles are bounded and all of them lead here.  Where sums are sent: everybody is set up.)
    __syncwarp();
    if constexpr (PUSH) {
      if (warp < 2) cluster_wait();
    } else {
      if (warp < 2) {
        cluster_arrive();
        cluster_wait();
        cluster_arrive();
      }
      cluster_wait();
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, alloc_cols);
  }
  if (threadIdx.x == 0 && g.stamp) stamp_max(g.stamp + 3);
  if constexpr (PUSH) {
    // All that is sent to this CTA has arrived, or it has given up: then it waits until the others are through (threads that
    // have left count as such), since its shared memory has to be there while they may still send to it.
    if (*reinterpret_cast<volatile uint32_t *>(&ctl->abort_flag) != 0) {
      __syncwarp();
      cluster_arrive();
      cluster_wait();
    }
  }
}

static size_t gemm_smem_bytes(int stages, int planes, int Mc) {
  return (size_t)stages * (kWBytes + planes * Mc * kBlockK * 2) + sizeof(GemmSmemCtl);
}

int gemm_pick_stages(int planes, int Mc, size_t smem_budget) {
  int s = kMaxStages;
  while (s > 2 && gemm_smem_bytes(s, planes, Mc) > smem_budget) --s;
  return s;
}

template <int EPI, bool PUSH = false>
static cudaError_t launch_one(const CUtensorMap &tw, const CUtensorMap &ta, const GemmArgs &g, dim3 grid,
                              size_t smem, cudaStream_t st, bool pdl) {
  static PerDeviceOnce once;
  int dev_ = -1;
  if (once.needed(&dev_)) {
    cudaError_t e = cudaFuncSetAttribute(gemm_ws_kernel<EPI, PUSH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         227 * 1024);
    if (e != cudaSuccess) return e;
    once.done(dev_);
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(192);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  int n = 0;
  if (grid.y > 1) {
    at[n].id = cudaLaunchAttributeClusterDimension;
    at[n].val.clusterDim.x = 1;
    at[n].val.clusterDim.y = grid.y;
    at[n].val.clusterDim.z = 1;
    ++n;
  }
  if (pdl) {
    at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
  }
  cfg.attrs = at;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, gemm_ws_kernel<EPI, PUSH>, tw, ta, g);
}

// (asked about a kernel without tensor memory: for one with it the occupancy call answers one CTA per SM)
__global__ void __launch_bounds__(192) cluster_probe_kernel(float *p) {
  extern __shared__ float s[];
  if (p) p[threadIdx.x] = s[threadIdx.x];
}
int gemm_max_clusters(int cluster, size_t smem_budget) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(1, cluster);
  cfg.blockDim = dim3(192);
  cfg.dynamicSmemBytes = smem_budget;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1;
  at[0].val.clusterDim.y = cluster;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaFuncSetAttribute(cluster_probe_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, cluster_probe_kernel, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

cudaError_t launch_gemm(int epi, const CUtensorMap &tw, const CUtensorMap &ta, GemmArgs g, int cluster,
                        size_t smem_budget, cudaStream_t st, bool pdl) {
  g.stages = gemm_pick_stages(g.planes, g.Mc, smem_budget);
  size_t smem = gemm_smem_bytes(g.stages, g.planes, g.Mc);
  const bool split = epi == EPI_QKV || epi == EPI_RESID;
  // Few rows: a CTA's sums go straight to the CTAs that finish the rows, 4 bytes per lane, counted by a barrier there, instead of
  // being fetched from it: one way through the cluster and no barriers of the cluster at the end (8B shape, one row: 76.4 -> 74.8
  // us per layer).  By 33 rows the small stores cost more than that (QKV of the 1B shape 5.1 -> 6.0 us, at 76 rows 8.1 -> 9.5).
  // They lie in what the ring leaves of the budget: with two planes that holds the rows of all steps of up to 16, but for 6 to 8 with
  // clusters of five and 8 with clusters of seven (two rows to a CTA beside boxes of eight), with one plane a row to a CTA.
  const size_t inbox = (size_t)cluster * ((g.M + cluster - 1) / cluster) * kTileN * 4;
  const bool push = split && cluster > 1 && g.M <= kPushRows && smem + inbox <= smem_budget;
  if (push) smem += inbox;
  if (g.N % kTileN || g.M > g.Mc || g.Mc % 8 || (g.planes * g.Mc) % 16 || cluster < 1 || cluster > (split ? 8 : 1) ||
      cluster > g.n_kblocks || g.stages * (kWBytes + g.planes * g.Mc * kBlockK * 2) < g.Mc * kTileN * 4)
    return cudaErrorInvalidValue;
  const dim3 grid(g.N / kTileN, cluster);
  switch (epi) {
    case EPI_QKV: return push ? launch_one<EPI_QKV, true>(tw, ta, g, grid, smem, st, pdl) : launch_one<EPI_QKV>(tw, ta, g, grid, smem, st, pdl);
    case EPI_RESID: return push ? launch_one<EPI_RESID, true>(tw, ta, g, grid, smem, st, pdl) : launch_one<EPI_RESID>(tw, ta, g, grid, smem, st, pdl);
    case EPI_SWIGLU: return launch_one<EPI_SWIGLU>(tw, ta, g, grid, smem, st, pdl);
    case EPI_LOGITS: return launch_one<EPI_LOGITS>(tw, ta, g, grid, smem, st, pdl);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace ts
