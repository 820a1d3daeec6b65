// Paged grouped-query attention of the verify chunk on the 5th-generation tensor cores, as a kernel of its own.
//
// One unit = (128-row tile of packed (position, query head) rows, kv head, run of KV positions); a CTA walks its units one
// after the other (tensor memory, barriers and the K/V ring are set up once and the ring keeps running across units).
//   warp 8   K/V producer: TMA loads of 64-position blocks straight from the pages (5-d tensor map over the pool)
//   warp 9   tensor memory allocation + tcgen05.mma issue:  S = Q K^T  (the unit's queries sit in tensor memory as
//            the row operand -- re-reading a 128-row query tile from shared memory for every 64-position block was
//            what bounded the kernel -- the K block K-major in shared memory, 128 x 64 fp32 result in tensor
//            memory), then  O += P V  with P read from tensor memory (fp16) and the V block read MN-major from
//            the same [position][64 elements] image K uses
//   warps 0..3, 4..7   two softmax groups, one row per thread: group 0 takes the unit's even blocks, group 1 the odd ones,
//            each with a reference maximum, a sum and output sums in tensor memory of its own, put together at the unit's
//            end.  Maximum over the block's 64 scores, P = exp2(S - reference maximum) written over the scores as an fp16
//            (value, rounding remainder) pair -- the second product adds both, so the 11 bits of fp16 do not limit the
//            weights (a single fp16 P was the largest error of the whole step).  The reference maximum follows the
//            running one in steps, and only then is the row of sums multiplied down
// A block is 1024 cycles of tensor-core work (24 instructions: both planes of Q and of P) and about 950 of softmax by one
// warp per scheduler, latency on latency; with one group the two alternated and a block took 2000 cycles, with two the
// one's softmax runs under the other's products: 1440 (four sessions with 64 rows each: from 8192 to 16384 tokens 62.1 -> 110.1
// us for 55.3 blocks more per SM, at the 1660 MHz that the power cap left beside it; at head_dim 64 37.5 -> 67.4 at 1965 MHz,
// 1060 cycles).  The rest of a launch, 14 us (7 at head_dim 64), is its CTAs' one or two units' set-up, first loads and way
// out.  What is left above 1024 is the issuing warp: an instruction is taken
// only when the ones before it are nearly done, so all that the warp does between two blocks leaves the tensor cores idle.
// Four sessions of 8192 tokens with 64 rows each: 81 -> 70 us per launch when the groups came; sixteen ragged ones: 114 -> 92.  (Measured and
// slower: an issuing warp per group, 86 and 114 us; exponentials before the block's maximum is known, 75 and 103.)
// Each unit writes an un-normalised partial output with its (max, sum); attn_merge_kernel adds a row's units.
// Every wait is bounded; on expiry the CTA records an error word and leaves through the normal exit.
#include <cuda_fp16.h>

#include <algorithm>

#include "kernels.h"
#include "schedule.h"

namespace ts {

static constexpr int kAttnRows = 128;   // packed rows per unit
static constexpr long long kMergeManyRows = 8192;   // (row, query head) pairs from which the merge takes several rows per warp
static constexpr int kAttnBlk = 64;     // kv positions per block
// K/V blocks in the ring (three are held by issued products, the rest are in flight): 192 KB of shared memory for
// either head width.  More than half of an SM's shared memory on purpose: a CTA takes all 512 columns of tensor memory,
// so a second one on the same SM would sit in its allocation until the first is done while other SMs stay idle.  With six
// stages of 16 KB (head_dim 64) the 128 CTAs of a 1B-shaped step were placed two to an SM: 13.5 us per launch at 4096
// tokens of context, 7 of them spent in that wait; with twelve stages 7.9 us (eight ragged sessions: 31.2 -> 15.3 us).
__host__ __device__ constexpr int kv_stages(int hd) { return hd == 64 ? 12 : 6; }
static constexpr int kMaxKvStages = 12;
static constexpr int kTcThreads = 320;
static constexpr int kStageBytes = 2048;   // per worker warp: 32 query rows x 64 bytes on their way to a row per thread (head_dim 64)
static constexpr int kWorkerWarps = 8, kProducerWarp = 8, kMmaWarp = 9;

struct __align__(16) AttnCtl {
  uint64_t kv_full[kMaxKvStages], kv_empty[kMaxKvStages], q_full;
  uint64_t s_full[2], p_full[2], pv_done[2];   // [2]: one per softmax group
  uint32_t tmem_base;
  // (reference maximum, sum) of each group's part of a row.  Two sets, for the CTA's units in turn: in a unit of one block
  // group 1 waits for nothing before it writes its (nothing), so a set may be written again only after the meeting of the
  // unit in between, which group 0 comes to when it has read this one.
  float2 ml[2][2][kAttnRows];
};

__device__ __forceinline__ bool worker_all(bool ok) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.and.pred q, 1, 256, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)ok)
      : "memory");
  return r != 0;
}
__device__ __forceinline__ bool mbar_wait_err(uint32_t bar, uint32_t parity, const int *err) {
  uint64_t t0 = 0;
  for (uint32_t it = 0;; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 255u) == 255u) {
      if (*reinterpret_cast<const volatile int *>(err) != 0) return false;
      const uint64_t now = global_timer_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > 2000000000ull) return false;
      __nanosleep(32);
    }
  }
}

// a unit with what follows from it
struct UnitInfo {
  int kh, slot, G;
  int r_beg, row0, rows_here, len;
  int pos_beg, pos_end, nblk;
};
__device__ __forceinline__ UnitInfo attn_unit_info(const AttnTcArgs &a, int u) {
  const int4 lo = *reinterpret_cast<const int4 *>(a.units + u), hi = *(reinterpret_cast<const int4 *>(a.units + u) + 1);
  UnitInfo t;
  t.r_beg = lo.y;
  t.row0 = lo.z;
  t.rows_here = lo.w;
  t.kh = hi.x & 0xFFFF;
  t.slot = hi.x >> 16;
  t.pos_beg = hi.y;
  t.pos_end = hi.z;
  t.len = hi.w;
  t.G = a.Hq / a.Hkv;
  if (!ts_in_range(a.in.ck, CHK_UNIT, lo.x, a.in.B) || !ts_in_range(a.in.ck, CHK_UNIT, t.slot, a.n_slots) ||
      !ts_in_range(a.in.ck, CHK_UNIT, t.kh, a.Hkv) || !ts_in_range(a.in.ck, CHK_UNIT, t.r_beg, a.in.M)) {
    // (debug build: the failed check is on record; go on with indices that are in range)
    t.slot = t.kh = t.r_beg = t.rows_here = 0;
  }
  t.nblk = t.pos_end > t.pos_beg ? (t.pos_end - t.pos_beg + kAttnBlk - 1) / kAttnBlk : 0;
  return t;
}

// tensor-memory columns
static constexpr int kColS = 0;      // one buffer of 64 columns per group: the scores, then in their place the probabilities as
                                     // fp16 pairs -- 32 columns of values, 32 of rounding remainders
static constexpr int kColQ = 128;    // the unit's queries, fp16 pairs: head_dim / 2 columns of values, then as many of remainders
static constexpr int kColO = 256;    // the output sums: head_dim columns per group (the second group's at + 128)
static constexpr float kRescaleStep = 8.f;   // the reference maximum follows the running one in steps of 2^8

// 2^x for x <= 0 (and 0 for -inf); tiny results flush to zero
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float y;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
  return y;
}
__device__ __forceinline__ uint32_t pack_h2(float x, float y) {
  __half2 v = __floats2half2_rn(x, y);
  return *reinterpret_cast<uint32_t *>(&v);
}

// Worker side of one unit.  Thread <-> row (tensor-memory lane q*32 + lane) of one of the two groups: it takes the row
// maximum over a block's 64 scores, writes the 64 probabilities over them as fp16 pairs and, rarely, rescales the row's
// output sums.  `cnt` counts this group's blocks over all units of this CTA (barrier parities come from it), `set` alternates
// over the CTA's units that have blocks (see AttnCtl::ml).
template <int HD>
__device__ __forceinline__ bool attn_unit_workers(const AttnTcArgs &a, AttnCtl *ctl, const UnitInfo &t, uint32_t tmem_base,
                                                  int grp, int q, int lane, uint32_t stg, uint32_t &cnt, uint32_t &set, bool &waited,
                                                  const int *err) {
  const int row = q * 32 + lane;      // row of the tile
  const int pr = t.row0 + row;        // packed row of the sequence
  const bool valid = row < t.rows_here;
  const int j = valid ? pr / t.G : 0, gq = valid ? pr % t.G : 0;
  const size_t ob = ((size_t)(t.r_beg + j) * a.Hq + t.kh * t.G + gq) * a.n_slots + t.slot;
  // (a step input like the unit tables: read before the dependency wait)
  const unsigned long long anc = ((unsigned long long)a.in.anc[2 * (t.r_beg + j) + 1] << 32) | a.in.anc[2 * (t.r_beg + j)];
  // head_dim 64: the queries come through a staging buffer per warp, 64 bytes of each of 32 rows at a time, so that a load
  // instruction touches eight rows in 64-byte pieces instead of 32 rows in 32-byte ones (1B shape, steps of 8 and 33 rows:
  // 748 -> 739 us, 967 -> 951; at head_dim 128 the loads of a thread's own row are as quick, and the staging's registers
  // spill).  This lane's part: rows 8 p + lane / 4 of the warp's 32 (their (row, query head) number, or -1), 16-byte piece
  // lane % 4.  Row r's piece s lies at slot s ^ (r / 2 % 4): no bank conflicts either way.
  constexpr bool kStaged = HD == 64;
  int rq[4];
  if constexpr (kStaged) {
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const int R = q * 32 + 8 * p + (lane >> 2), x = t.row0 + R;
      rq[p] = R < t.rows_here ? (t.r_beg + x / t.G) * a.Hq + t.kh * t.G + x % t.G : -1;
    }
  }
  // the rotated queries come from the previous kernel; everything above was on the device before the step began
  if (!waited) {
    pdl_wait();
    waited = true;
    if (threadIdx.x == 0) stamp_waited(a.stamp);
  }
  if (t.nblk == 0) {   // no position in this unit: mark its slot empty
    if (valid && grp == 0) a.attn_ml[ob] = make_float2(-INFINITY, 0.f);
    return true;
  }
  // ---- stage Q into tensor memory: the score product reads its row operand there (thread <-> row, an fp16 pair
  // per column; group 0 the values, group 1 the rounding remainders), so per block only the keys and values come
  // through shared memory.  Every score product of the CTA's previous unit has completed (both groups had read their last
  // scores when they met at its end), so the columns may be overwritten.
  const uint32_t tq = tmem_base + ((uint32_t)(q * 32) << 16);
  {
    // (either way all loads are issued before the first use: one round trip to L2)
    if constexpr (kStaged) {
      const __half *src = grp ? a.q_lo : a.q;
      const int piece = lane & 3;
      auto slot_of = [&](int r, int s) { return (uint32_t)((s ^ ((r >> 1) & 3)) << 4); };
      uint4 v[HD / 32][4];
#pragma unroll
      for (int c = 0; c < HD / 32; ++c)
#pragma unroll
        for (int p = 0; p < 4; ++p)
          v[c][p] = rq[p] >= 0 ? *reinterpret_cast<const uint4 *>(src + (size_t)rq[p] * HD + c * 32 + piece * 8) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
      for (int c = 0; c < HD / 32; ++c) {
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          const int R = 8 * p + (lane >> 2);
          st_shared_v4(stg + R * 64 + slot_of(R, piece), v[c][p].x, v[c][p].y, v[c][p].z, v[c][p].w);
        }
        __syncwarp();
        uint32_t r[16];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const uint4 w = ld_shared_v4(stg + lane * 64 + slot_of(lane, s));
          r[4 * s] = w.x; r[4 * s + 1] = w.y; r[4 * s + 2] = w.z; r[4 * s + 3] = w.w;
        }
        __syncwarp();
        tmem_st16(tq + kColQ + grp * (HD / 2) + c * 16, r);
      }
    } else {
      const __half *src = (grp ? a.q_lo : a.q) + ((size_t)(t.r_beg + j) * a.Hq + t.kh * t.G + gq) * HD;
      // all loads are issued before the first use: one round trip to L2, where the previous kernel has just written the
      // rows (32 bytes per lane and load: the lanes of a warp read 32 different rows)
      uint32_t v[HD / 2];
      if (valid) {
#pragma unroll
        for (int c = 0; c < HD / 16; ++c) ld_global_v8(src + c * 16, &v[c * 8]);
      } else {
#pragma unroll
        for (int c = 0; c < HD / 2; ++c) v[c] = 0u;
      }
#pragma unroll
      for (int c4 = 0; c4 < HD / 32; ++c4) {
        uint32_t r[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) r[e] = v[c4 * 16 + e];
        tmem_st16(tq + kColQ + grp * (HD / 2) + c4 * 16, r);
      }
    }
    tmem_wait_st();
  }
  tc_fence_before();
  __syncwarp();
  if (lane == 0) mbar_arrive(smem_u32(&ctl->q_full));

  // Visibility: the whole cache, and of the chunk the rows named by this row's mask (itself and its ancestors in
  // the draft tree; in a chain, rows 0..j), up to the end of this unit.
  const int lim_all = min(t.len, t.pos_end) - 1;   // every row sees every position up to here
  const float scale = rsqrtf((float)HD) * 1.4426950408889634f;
  // The output sums stay in tensor memory: every product P V adds to them.  Probabilities are taken against a
  // reference maximum m_ref that follows the running maximum lazily: only when a block's maximum exceeds it by
  // more than kRescaleStep (in the log2 domain) is the row of sums multiplied down and m_ref raised, so in most
  // blocks the softmax thread never touches the sums.  Until then probabilities may reach 2^kRescaleStep: well
  // inside fp16, and the sums are fp32.
  float m_ref = -INFINITY, l_run = 0.f;
  bool ok = true;
  const uint32_t colS = tq + kColS + grp * 64, colO = tq + kColO + grp * 128;

  for (int b = grp; b < t.nblk; b += 2, ++cnt) {
    if (ok && !mbar_wait_err(smem_u32(&ctl->s_full[grp]), cnt & 1, err)) { ok = false; atomicCAS((int *)err, 0, DEV_TIMEOUT_TMEM); }
    tc_fence_after();
    const int p_base = t.pos_beg + b * kAttnBlk;
    float sc[64];
    {
      uint32_t r0[16], r1[16], r2[16], r3[16];
      tmem_ld16(colS, r0);
      tmem_ld16(colS + 16, r1);
      tmem_ld16(colS + 32, r2);
      tmem_ld16(colS + 48, r3);
      tmem_wait_ld();
#pragma unroll
      for (int e = 0; e < 16; ++e) {
        sc[e] = __uint_as_float(r0[e]); sc[16 + e] = __uint_as_float(r1[e]);
        sc[32 + e] = __uint_as_float(r2[e]); sc[48 + e] = __uint_as_float(r3[e]);
      }
    }
    // a block every row sees whole needs no mask (all but the last blocks of a sequence's last unit)
    if (p_base + kAttnBlk - 1 > lim_all) {
      // bit e of `vis`: position p_base + e is visible to this row (cache positions all, chunk rows by the mask,
      // nothing at or past the unit's end)
      const int rel0 = p_base - t.len;                 // chunk row of the block's first position (negative: cache)
      unsigned long long vis;
      if (rel0 >= 0) vis = rel0 < 64 ? anc >> rel0 : 0ull;
      else if (rel0 > -64) vis = (anc << (-rel0)) | ((1ull << (-rel0)) - 1ull);
      else vis = ~0ull;
      const int n_in = t.pos_end - p_base;             // positions of the block inside the unit
      if (n_in < 64) vis &= n_in > 0 ? (1ull << n_in) - 1ull : 0ull;
      const uint32_t vlo = (uint32_t)vis, vhi = (uint32_t)(vis >> 32);
#pragma unroll
      for (int e = 0; e < 32; ++e) {
        sc[e] = (vlo >> e) & 1u ? sc[e] : -INFINITY;
        sc[32 + e] = (vhi >> e) & 1u ? sc[32 + e] : -INFINITY;
      }
    }
    float mx0 = -INFINITY, mx1 = -INFINITY, mx2 = -INFINITY, mx3 = -INFINITY;
#pragma unroll
    for (int e = 0; e < 64; e += 8) {   // three-input maxima: half the instructions of pairwise ones
      mx0 = max3(mx0, sc[e], sc[e + 1]); mx1 = max3(mx1, sc[e + 2], sc[e + 3]);
      mx2 = max3(mx2, sc[e + 4], sc[e + 5]); mx3 = max3(mx3, sc[e + 6], sc[e + 7]);
    }
    // block maximum in the log2 domain: scores times log2(e)/sqrt(head_dim), folded into one multiply-add per score
    const float m_blk = fmaxf(fmaxf(mx0, mx1), fmaxf(mx2, mx3)) * scale;
    const bool raise = m_blk > m_ref + kRescaleStep;   // (also the first finite maximum: m_ref starts at -inf)
    const float m_old = m_ref;
    if (raise) m_ref = m_blk;
    const float ref = (m_ref == -INFINITY) ? 0.f : m_ref;
    // Multiplying the sums down needs the group's previous product complete, and it is: it was issued before this block's
    // scores, whose commit covers everything issued before it.
    float f = 1.f;
    if (b > grp && __any_sync(0xffffffffu, raise)) {     // tensor-memory accesses are warp-wide: lanes that stay use f = 1
      if (raise) f = ex2_approx(m_old - ref);            // exp2(-inf) = 0: nothing was summed before the first finite maximum
#pragma unroll
      for (int i = 0; i < HD / 32; ++i) {
        uint32_t r0[16], r1[16];
        tmem_ld16(colO + i * 32, r0);
        tmem_ld16(colO + i * 32 + 16, r1);
        tmem_wait_ld();
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          r0[e] = __float_as_uint(__uint_as_float(r0[e]) * f);
          r1[e] = __float_as_uint(__uint_as_float(r1[e]) * f);
        }
        tmem_st16(colO + i * 32, r0);
        tmem_st16(colO + i * 32 + 16, r1);
      }
    }
    const float2 scale2 = make_float2(scale, scale), nref2 = make_float2(-ref, -ref), minus1 = make_float2(-1.f, -1.f);
    float2 sum0 = make_float2(0.f, 0.f), sum1 = sum0;
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {   // 32 scores at a time: 16 columns of values, 16 of remainders
      uint32_t pk[16], pl[16];
#pragma unroll
      for (int e = 0; e < 16; ++e) {
        float2 x = fma2(make_float2(sc[32 * hh + 2 * e], sc[32 * hh + 2 * e + 1]), scale2, nref2);
        x.x = ex2_approx(x.x);
        x.y = ex2_approx(x.y);
        if (e & 1) sum1 = add2(sum1, x);
        else sum0 = add2(sum0, x);
        const __half2 h = __floats2half2_rn(x.x, x.y);
        pk[e] = *reinterpret_cast<const uint32_t *>(&h);
        const float2 rest = fma2(__half22float2(h), minus1, x);   // x - h, exact
        pl[e] = pack_h2(rest.x, rest.y);
      }
      tmem_st16(colS + 16 * hh, pk);
      tmem_st16(colS + 32 + 16 * hh, pl);
    }
    sum0 = add2(sum0, sum1);
    l_run = l_run * f + (sum0.x + sum0.y);
    tmem_wait_st();
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&ctl->p_full[grp]));
    // (no CTA-wide barrier per block: a failed wait has set the error word, which ends every other wait)
  }
  // the group's last product; its earlier ones are known complete (see above), so a parity wait is enough
  const bool any = t.nblk > grp;
  if (any && ok && !mbar_wait_err(smem_u32(&ctl->pv_done[grp]), (cnt - 1) & 1, err)) { ok = false; atomicCAS((int *)err, 0, DEV_TIMEOUT_TMEM); }
  tc_fence_after();
  float2(*ml)[kAttnRows] = ctl->ml[set];
  set ^= 1u;
  ml[grp][row] = make_float2(m_ref, l_run);
  tc_fence_before();
  if (!worker_all(ok)) return false;
  tc_fence_after();

  // ---- partial result of this unit: un-normalised output, its reference maximum (log2 domain), sum.  Each thread puts
  // half of its row's output together from both groups' sums.
  {
    const float2 m0 = ml[0][row], m1 = ml[1][row];
    const float m = fmaxf(m0.x, m1.x);
    const float w0 = m0.x == -INFINITY ? 0.f : ex2_approx(m0.x - m), w1 = m1.x == -INFINITY ? 0.f : ex2_approx(m1.x - m);
    float *dst = a.attn_o + ob * HD + grp * (HD / 2);
    if (valid && grp == 0) a.attn_ml[ob] = make_float2(m, m0.y * w0 + m1.y * w1);
    const uint32_t src = tq + kColO + grp * (HD / 2);
    const bool both = t.nblk > 1;   // (else group 1's sums were never started)
#pragma unroll
    for (int i = 0; i < HD / 32; ++i) {
      uint32_t r0[16], r1[16];
      tmem_ld16(src + i * 16, r0);      // (warp-wide: rows past the tile's end read too, and write nothing)
      if (both) tmem_ld16(src + 128 + i * 16, r1);
      tmem_wait_ld();
#pragma unroll
      for (int e = 0; e < 16; ++e)
        r0[e] = __float_as_uint(__uint_as_float(r0[e]) * w0 + (both ? __uint_as_float(r1[e]) * w1 : 0.f));
      if (valid) {   // whole 32-byte sectors per lane: the lanes of a warp write 32 different rows
        st_global_v8(dst + i * 16, r0);
        st_global_v8(dst + i * 16 + 8, r0 + 8);
      }
    }
  }
  // (The output sums are in registers / on their way to memory; the next unit's first products, which overwrite them, wait
  // for its queries, which this warp stages next.)
  return true;
}

template <int HD>
__global__ void __launch_bounds__(kTcThreads, 1) attn_tc_kernel(const __grid_constant__ AttnTcArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  constexpr uint32_t kKvBytes = 2u * kAttnBlk * HD * 2, kHalves = HD / 64;
  constexpr int kKvStages = kv_stages(HD);
  AttnCtl *ctl = reinterpret_cast<AttnCtl *>(smem + kKvStages * kKvBytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int *err = a.err;

  if (threadIdx.x == 0) {
    for (int b = 0; b < kKvStages; ++b) {
      mbar_init(smem_u32(&ctl->kv_full[b]), 1);
      mbar_init(smem_u32(&ctl->kv_empty[b]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&ctl->s_full[b]), 1);
      mbar_init(smem_u32(&ctl->p_full[b]), 4);
      mbar_init(smem_u32(&ctl->pv_done[b]), 1);
    }
    mbar_init(smem_u32(&ctl->q_full), kWorkerWarps);   // one arrival per worker warp
    fence_barrier_init();
  }
  if (warp == kMmaWarp) {
    tmem_alloc(smem_u32(&ctl->tmem_base), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = ctl->tmem_base;
  if (threadIdx.x == 0) stamp_min(a.stamp);
  pdl_launch_dependents();   // (this CTA holds its tensor memory; the dependent waits for this kernel's end anyway)
  // The step's integer inputs were copied in before the step's first kernel started, so they may be read here.
  // The three roles walk this CTA's units as three loops coupled only by the barriers, whose phases are counted over all
  // blocks (`gb`) and units (`un`) of the CTA.
  const int u_beg = a.cta_unit[blockIdx.x], u_end = a.cta_unit[blockIdx.x + 1];

  if (warp == kProducerWarp) {
    // ---------------------------------------------------------------- K/V producer
    // (the whole warp walks the loops and the waits; an elected lane issues a block's sixteen copies -- a lone lane
    // in a divergent branch needs about 50 cycles per copy instruction, more than half of a block's time)
    {
      const uint64_t pol = policy_evict_first();
      uint32_t gb = 0;
      bool waited = false, ok = true;
      for (int u = u_beg; u < u_end && ok; ++u) {
        const UnitInfo t = attn_unit_info(a, u);
        const int32_t *btab = a.in.block_tab + (size_t)a.units[u].seq * a.in.pages_per_seq;
        const int ready = a.ready_len >= 0 ? a.ready_len : t.len;
        for (int b = 0; b < t.nblk; ++b, ++gb) {
          // blocks wholly inside the cache of earlier steps do not depend on the previous kernel: the ring is filled
          // with them before the dependency wait; the chunk's own K/V rows come from the previous kernel
          if (!waited && (gb >= (uint32_t)kKvStages || t.pos_beg + (b + 1) * kAttnBlk > ready)) { pdl_wait(); waited = true; }
          const uint32_t st = gb % kKvStages;
          if (gb >= (uint32_t)kKvStages &&
              !__all_sync(0xffffffffu, mbar_wait_err(smem_u32(&ctl->kv_empty[st]), ((gb / kKvStages) & 1) ^ 1, err))) {
            if (lane == 0) atomicCAS(a.err, 0, DEV_TIMEOUT_EMPTY);
            ok = false;
            break;
          }
          const uint32_t bar = smem_u32(&ctl->kv_full[st]);
          uint8_t *sK = smem + st * kKvBytes, *sV = sK + kAttnBlk * HD * 2;
          // lane pg looks its page up (a page past the unit's end is never visible: the last visible page is loaded
          // again instead); the elected lane gets the four ids by shuffle
          int page = 0;
          if (lane < kAttnBlk / 16) {
            const int pos = min(t.pos_beg + b * kAttnBlk + lane * 16, t.pos_end - 1);
            page = btab[pos >> 4];
            if (!ts_in_range(a.in.ck, CHK_PAGE_ATTN, page, a.in.ck.max_pages)) page = 0;
          }
          int pages[kAttnBlk / 16];
#pragma unroll
          for (int pg = 0; pg < kAttnBlk / 16; ++pg) pages[pg] = __shfl_sync(0xffffffffu, page, pg);
          if (elect_one()) {
            mbar_expect_tx(bar, kKvBytes);
#pragma unroll
            for (int pg = 0; pg < kAttnBlk / 16; ++pg) {
#pragma unroll
              for (int hh = 0; hh < (int)kHalves; ++hh) {
                const uint32_t off = hh * (kAttnBlk * 128) + pg * 2048;
                tma_load_5d(smem_u32(sK + off), a.map_kv, hh * 64, 0, t.kh, pages[pg], 2 * a.layer, bar, pol);
                tma_load_5d(smem_u32(sV + off), a.map_kv, hh * 64, 0, t.kh, pages[pg], 2 * a.layer + 1, bar, pol);
              }
            }
          }
          __syncwarp();
        }
      }
    }
  } else if (warp == kMmaWarp) {
    // ---------------------------------------------------------------- MMA issue
    // The whole warp walks the loops and the waits together; one elected lane issues a block's tensor-core instructions
    // and commits (the loop state is then the same in every lane, which lets the compiler keep descriptors and addresses
    // in uniform registers: a lone lane in a divergent branch issued an instruction every ~50 cycles).
    {
      const uint32_t idesc_qk = umma_idesc_f16(kAttnRows, kAttnBlk, 0);
      const uint32_t idesc_pv = umma_idesc_f16(kAttnRows, HD, 1);
      const uint32_t sKV = smem_u32(smem);
      bool ok = true;
      uint32_t gb = 0, un = 0, par = 0;   // par: bit g = parity of group g's blocks so far
      // a wait that ran out in one lane ends the loops of all lanes together (elect.sync names the full warp)
      auto wait_all = [&](uint32_t bar, uint32_t parity) -> bool {
        return __all_sync(0xffffffffu, mbar_wait_err(bar, parity, err));
      };
      // S = Q K^T + Q_lo K^T for the CTA's block bi into group g's buffer: the remainder plane of the queries goes through
      // the same keys into the same sums; the queries are read from tensor memory (8 columns = 16 elements per
      // instruction).  The buffer is free: the product that read the group's previous probabilities was issued before.
      auto qk = [&](uint32_t g, uint32_t bi) {
        const uint64_t dk = umma_desc_sw128(sKV + (bi % kKvStages) * kKvBytes);
        const uint32_t colS = tmem_base + kColS + g * 64;
#pragma unroll
        for (int pl = 0; pl < 2; ++pl)
#pragma unroll
          for (int hh = 0; hh < (int)kHalves; ++hh)
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              umma_f16_ts(colS, tmem_base + kColQ + pl * (HD / 2) + hh * 32 + kk * 8, dk + hh * (kAttnBlk * 128 / 16) + 2 * kk,
                          idesc_qk, (pl | hh | kk) != 0 ? 1u : 0u);
        umma_commit(smem_u32(&ctl->s_full[g]));
      };
      // O (+)= P V for block b of the unit, the CTA's block bi; a group's first block of a unit starts its sums afresh
      auto pv = [&](int b, uint32_t bi) {
        const uint32_t vst = bi % kKvStages, g = b & 1;
        const uint32_t colO = tmem_base + kColO + g * 128, colP = tmem_base + kColS + g * 64;
        const uint64_t dv = umma_desc_sw128_mn(sKV + vst * kKvBytes + kAttnBlk * HD * 2, kAttnBlk * 128);
#pragma unroll
        for (int ks = 0; ks < kAttnBlk / 16; ++ks) {   // 16 positions per instruction: values, then remainders
          umma_f16_ts(colO, colP + ks * 8, dv + ks * (2048 / 16), idesc_pv, (b > 1 || ks != 0) ? 1u : 0u);
          umma_f16_ts(colO, colP + 32 + ks * 8, dv + ks * (2048 / 16), idesc_pv, 1u);
        }
        umma_commit(smem_u32(&ctl->pv_done[g]));
        umma_commit(smem_u32(&ctl->kv_empty[vst]));
      };
      auto wait_kv = [&](uint32_t bi) { return wait_all(smem_u32(&ctl->kv_full[bi % kKvStages]), (bi / kKvStages) & 1); };
      // Issue order within a unit: S(0), S(1), then for every block b: O += P(b) V(b), S(b + 2).  While one group works
      // on its scores the other's products run.
      for (int u = u_beg; u < u_end && ok; ++u) {
        const UnitInfo t = attn_unit_info(a, u);
        if (t.nblk == 0) continue;
        ok = wait_all(smem_u32(&ctl->q_full), un & 1) && wait_kv(gb);
        ++un;
        tc_fence_after();
        if (ok && elect_one()) qk(0, gb);
        __syncwarp();
        if (ok && t.nblk > 1) {
          ok = wait_kv(gb + 1);
          tc_fence_after();
          if (ok && elect_one()) qk(1, gb + 1);
          __syncwarp();
        }
        for (int b = 0; ok && b < t.nblk; ++b, ++gb) {
          // (the keys of block b + 2 first: they are long there, and nothing comes between the block's products then)
          const bool more = b + 2 < t.nblk;
          // (both barriers are looked at together: what this warp does between two issues leaves the tensor cores idle)
          const uint32_t kv2 = gb + (more ? 2 : 0), bar_kv = smem_u32(&ctl->kv_full[kv2 % kKvStages]), par_kv = (kv2 / kKvStages) & 1;
          const uint32_t bar_p = smem_u32(&ctl->p_full[b & 1]), par_p = (par >> (b & 1)) & 1;
          if (!__all_sync(0xffffffffu, mbar_try_wait(bar_kv, par_kv) & mbar_try_wait(bar_p, par_p)))
            ok = wait_all(bar_kv, par_kv) && wait_all(bar_p, par_p);
          par ^= 1u << (b & 1);
          tc_fence_after();
          if (ok && elect_one()) {
            pv(b, gb);
            if (more) qk(b & 1, gb + 2);
          }
          __syncwarp();
        }
      }
      if (!ok && lane == 0) atomicCAS(a.err, 0, DEV_TIMEOUT_FULL);
    }
  } else {
    // ---------------------------------------------------------------- workers
    uint32_t cnt = 0, set = 0;
    bool ok = true, waited = false;
    for (int u = u_beg; u < u_end && ok; ++u) {
      const UnitInfo t = attn_unit_info(a, u);
      ok = attn_unit_workers<HD>(a, ctl, t, tmem_base, warp >> 2, warp & 3, lane, smem_u32(ctl + 1) + warp * kStageBytes, cnt, set, waited, err);
    }
    if (!waited) pdl_wait();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
  if (threadIdx.x == 0 && a.stamp) stamp_max(a.stamp + 3);
}

// grid = (M / RW, Hq / 4), 4 warps: a warp adds the partial results of RW rows of one query head and emits the normalised
// rows as bf16 (hi[, lo]); lane i owns hd / 32 consecutive elements.  The (tile, kv head) has tile_slots units, all of them
// written (one the row sees nothing of carries sum 0 and gets weight 0).  Lane s turns slot s's (max, sum) into a weight;
// every lane loads its elements of all slots at once (one round trip to L2, 16 bytes per lane and slot) and adds them in
// slot order.  NS = compile-time bound on the number of slots.  (RW > 1 for many rows, where a row at a time is several
// waves of CTAs that each wait for a few round trips: 1024 rows of the 8B shape 29 us, four at a time 9.5.)
template <int NS, int VW, int RW>
__global__ void __launch_bounds__(128) attn_merge_kernel(const AttnTcArgs a) {
  if (threadIdx.x == 0) stamp_min(a.stamp_merge);
  pdl_launch_dependents();   // the dependent kernel waits for this one's end before touching its data
  const int m0 = blockIdx.x * RW, h = blockIdx.y * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  // (step inputs, on the device before the step's first kernel)
  const int G = a.Hq / a.Hkv;
  int nl[RW];
#pragma unroll
  for (int i = 0; i < RW; ++i) {
    nl[i] = 0;
    if (h < a.Hq && m0 + i < a.in.M) {
      const int meta = a.in.row_tile[m0 + i];
      nl[i] = a.tile_slots[((meta >> 6) + ((meta & 63) * G + h % G) / kAttnRows) * a.Hkv + h / G];
    }
    if (!ts_in_range(a.in.ck, CHK_LEAVES, nl[i], a.n_slots + 1)) nl[i] = 0;
  }
  pdl_wait();
  if (threadIdx.x == 0) stamp_waited(a.stamp_merge);
  if (h >= a.Hq) return;
  float2 ml[RW];
  float t[RW][NS][VW];
#pragma unroll
  for (int i = 0; i < RW; ++i) {
    const size_t base = ((size_t)(m0 + i) * a.Hq + h) * a.n_slots;
    ml[i] = lane < nl[i] ? a.attn_ml[base + lane] : make_float2(-INFINITY, 0.f);
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      const float *src = a.attn_o + (base + s) * a.hd + lane * VW;
      if constexpr (VW == 4) {
        const float4 v = ld_global_v4_if(src, s < nl[i]);
        t[i][s][0] = v.x; t[i][s][1] = v.y; t[i][s][2] = v.z; t[i][s][3] = v.w;
      } else {
        const float2 v = ld_global_v2_if(src, s < nl[i]);
        t[i][s][0] = v.x; t[i][s][1] = v.y;
      }
    }
  }
  __syncwarp();   // (no load may move past it: left to itself the compiler puts every load next to its use)
#pragma unroll
  for (int i = 0; i < RW; ++i) {
    const int m = m0 + i;
    if (m >= a.in.M) break;
    float mx = ml[i].y > 0.f ? ml[i].x : -INFINITY;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    float w = ml[i].y > 0.f ? exp2f(ml[i].x - mx) : 0.f;
    // the denominator: slot by slot in slot order (a shuffle tree would pair lanes differently as slots are added)
    float den = 0.f, num[VW];
#pragma unroll
    for (int e = 0; e < VW; ++e) num[e] = 0.f;
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      const float ws = __shfl_sync(0xffffffffu, w, s);
      const float ls = __shfl_sync(0xffffffffu, ml[i].y, s);
      den += ws * ls;
#pragma unroll
      for (int e = 0; e < VW; ++e) num[e] += ws * (ws != 0.f ? t[i][s][e] : 0.f);
    }
    const float inv = 1.f / den;
    __align__(8) __nv_bfloat16 hi[VW], lo[VW];
#pragma unroll
    for (int e = 0; e < VW; ++e) split_bf16(num[e] * inv, hi[e], lo[e]);
    const size_t col = (size_t)h * a.hd + lane * VW;
    const size_t ld = (size_t)a.Hq * a.hd;
    __nv_bfloat16 *o_hi = a.out + (size_t)m * ld + col, *o_lo = a.out + ((size_t)a.out_rows + m) * ld + col;
    if constexpr (VW == 4) {
      *reinterpret_cast<uint2 *>(o_hi) = *reinterpret_cast<const uint2 *>(hi);
      if (a.planes == 2) *reinterpret_cast<uint2 *>(o_lo) = *reinterpret_cast<const uint2 *>(lo);
    } else {
      *reinterpret_cast<uint32_t *>(o_hi) = *reinterpret_cast<const uint32_t *>(hi);
      if (a.planes == 2) *reinterpret_cast<uint32_t *>(o_lo) = *reinterpret_cast<const uint32_t *>(lo);
    }
  }
  if (threadIdx.x == 0 && a.stamp_merge) stamp_max(a.stamp_merge + 3);
}

template <int NS, int VW, int RW>
static cudaError_t launch_merge_pdl(const AttnTcArgs &a, cudaStream_t st) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((a.in.M + RW - 1) / RW, (a.Hq + 3) / 4);
  cfg.blockDim = dim3(128);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, attn_merge_kernel<NS, VW, RW>, a);
}

template <int VW>
static cudaError_t launch_merge(const AttnTcArgs &a, cudaStream_t st) {
  // four rows per warp where that still fills the SMs' warps about once
  const bool many = (long long)a.in.M * a.Hq >= kMergeManyRows;
  if (a.n_slots <= 2) return many ? launch_merge_pdl<2, VW, 4>(a, st) : launch_merge_pdl<2, VW, 1>(a, st);
  if (a.n_slots <= 4) return many ? launch_merge_pdl<4, VW, 4>(a, st) : launch_merge_pdl<4, VW, 1>(a, st);
  if (a.n_slots <= 8) return many ? launch_merge_pdl<8, VW, 2>(a, st) : launch_merge_pdl<8, VW, 1>(a, st);
  if (a.n_slots <= 16) return launch_merge_pdl<16, VW, 1>(a, st);
  return launch_merge_pdl<32, VW, 1>(a, st);
}

cudaError_t launch_attention_tc_merge(const AttnTcArgs &a, cudaStream_t st) {
  if (a.n_slots < 1 || a.n_slots > kAttnMaxSplits) return cudaErrorInvalidValue;
  return a.hd == 128 ? launch_merge<4>(a, st) : launch_merge<2>(a, st);
}

static size_t attn_tc_smem(int hd) {
  return 1024 + (size_t)kv_stages(hd) * 2 * kAttnBlk * hd * 2 + sizeof(AttnCtl) + (hd == 64 ? kWorkerWarps * kStageBytes : 0) + 64;
}

cudaError_t launch_attention_tc(const AttnTcArgs &a, cudaStream_t st) {
  static PerDeviceOnce once;
  int dev_ = -1;
  if (once.needed(&dev_)) {
    cudaError_t e = cudaFuncSetAttribute(attn_tc_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)attn_tc_smem(128));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(attn_tc_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)attn_tc_smem(64));
    if (e != cudaSuccess) return e;
    once.done(dev_);
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(a.n_ctas);
  cfg.blockDim = dim3(kTcThreads);
  cfg.dynamicSmemBytes = attn_tc_smem(a.hd);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return (a.hd == 128) ? cudaLaunchKernelEx(&cfg, attn_tc_kernel<128>, a) : cudaLaunchKernelEx(&cfg, attn_tc_kernel<64>, a);
}

}  // namespace ts
