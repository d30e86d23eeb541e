// Window scoring on the tensor cores (tcgen05 MMA, accumulator in TMEM, operands fed by TMA).
//
// Two kernels over one skeleton.  The work is the linear space of (virtual unit, key tile) pairs;
// it is cut into equal contiguous ranges, one per CTA, and at most one CTA per SM is launched, so
// a CTA streams a long run of key tiles through its TMA ring and pays its start-up once.  A
// virtual unit is a (batch, kv-head) unit, or for the statistics one half of its window rows when
// there are more than 256; its query rows stay resident in shared memory and are reloaded when
// the CTA's range crosses into the next virtual unit.
// Warp roles: four consumer warpgroups in two pairs read the accumulators out of TMEM (one TMEM
// lane per thread; pair p drains accumulator buffer p, each of its groups half of the columns), one
// warp is the TMA producer, one warp allocates TMEM and issues the MMAs.  What bounds both kernels is the
// exponentials, one per logit; see exp2.cuh.  32 units x 256 rows x 32768 keys: statistics 170 -> 140 thousand
// cycles (ncu, 92 -> 85 us at the clock the power limit leaves), votes 172 -> 142 (94 -> 86 us), with a share
// of the exponentials on the FMA pipe and the work between two jobs cut down; either alone gave little (the
// polynomial without the other change: 173 and 189 thousand cycles).  Every MMA has N = 256 where the shape allows
// it: with both operands in shared memory, narrower tiles are limited by operand fetch, not by the tensor pipe.
//
//   statistics (kVotes = false):  S = Q K^T, 128 query rows on the TMEM lanes, 256 keys per tile.
//       Thread r keeps the running (max, sum) of exp2(scale2 * s) over the keys row r may see
//       (causal inside the window).  Per-CTA partials are combined into the natural-log row LSE by
//       row_lse_from_parts_kernel.  Skipped altogether when the caller supplies the row LSE.
//   votes (kVotes = true):  S^T = K Q^T, 128 KEYS on the TMEM lanes and up to 256 query rows as
//       columns, so the vote of a key, sum over rows of exp2(scale2 * s - lse2[row]), is a
//       per-thread sum over the accumulator's columns: no cross-thread reduction and fp32
//       probabilities throughout.  The groups' halves go out as parts that the selection adds up.
//       Candidate keys (t < L - W) are seen by every window row, so this pass needs no mask.
#include <type_traits>

#include "exp2.cuh"
#include "internal.h"
#include "tc_common.cuh"

namespace calidrop {

namespace {

using namespace tc;

constexpr int kGroups = 4;  // consumer warpgroups (4 warps each), two pairs; pair p drains accumulator buffer p
constexpr int kProducerWarp = kGroups * 4;
constexpr int kMmaWarp = kGroups * 4 + 1;
constexpr int kThreads = kGroups * 128 + 64;
constexpr int kTmemCols = 512;  // two accumulators of 256 columns or four of 128
constexpr int kMaxBufs = 4;
constexpr int kMaxRows = 512;   // G * W handled by the tiles

// Where the partial statistics of a row lie: those of the CTAs whose tile range overlaps the row's virtual unit.
struct StatParts {
  const float2* part;   // [row][slot][n_part] (max, sum)
  int vu_per_unit, n_tiles, tiles_per_cta, max_slots, n_part;
  __device__ __forceinline__ const float2* of(int unit, int GW, int row, int* n) const {
    const int vu = unit * vu_per_unit + row / 256;
    const int first = (vu * n_tiles) / tiles_per_cta, last = ((vu + 1) * n_tiles - 1) / tiles_per_cta;
    *n = (last - first + 1) * n_part;
    return part + (size_t)(unit * GW + row) * max_slots * n_part;
  }
};

struct ScoreArgs {
  int Hq, G, W, L, n_cand, GW;
  int vu_per_unit;    // virtual units per (batch, kv-head) unit
  int vu_rows;        // window rows a virtual unit starts at: vu % vu_per_unit * vu_rows
  int n_blocks;       // row blocks (= accumulators) per key tile
  int block_rows;     // rows per block: 128 for the statistics, a multiple of 64 (<= 256) for the votes
  int n_tiles;        // key tiles per virtual unit
  int total_tiles;    // virtual units * n_tiles
  int tiles_per_cta;
  int stages;         // depth of the key-tile ring
  int lg_bufs;        // log2 of the accumulator count: two of 256 columns, or four of 128
  int max_slots;      // statistics: partial slots per row (CTAs that can share a virtual unit)
  float scale2;
  const float* row_lse;  // votes: natural-log LSE of every observation row [B, Hq, W]
  float* vote_parts;     // votes: out [part][units, n_cand], a part per (row block, column half)
  float2* stat_part;     // statistics: out [row][slot][2 or 4 groups] (max, sum) in the log2 domain
  // votes: the statistics' partials, combined here (StatParts::part null: row_lse is given)
  StatParts stats;
  float* lse_out;        // ... and the natural-log LSE for the calibration
  int lg_tpr;            // ... log2 of the threads that share a row
  unsigned* status;
  int clear_status;      // the first kernel of a call clears the error word
};

// sum of exp2 of 32 logits against one reference, four independent partial sums
__device__ __forceinline__ float sum_exp2_32(const uint32_t (&r)[32], f32x2 sc, f32x2 nr) {
  f32x2 s0 = 0ull, s1 = 0ull;
#pragma unroll
  for (int e = 0; e < 32; e += 4) {
    const f32x2 x0 = fma2(pack2(r[e], r[e + 1]), sc, nr), x1 = fma2(pack2(r[e + 2], r[e + 3]), sc, nr);
    s0 = add_exp2_pair<false>(s0, x0, e / 2);
    s1 = add_exp2_pair<false>(s1, x1, e / 2 + 1);
  }
  const float2 v = unpack2(add2(s0, s1));
  return v.x + v.y;
}

__device__ __forceinline__ float max_32(const uint32_t (&r)[32]) {
  float m0 = -INFINITY, m1 = -INFINITY, m2 = -INFINITY, m3 = -INFINITY;
#pragma unroll
  for (int e = 0; e < 32; e += 4) {
    m0 = fmaxf(m0, __uint_as_float(r[e + 0]));
    m1 = fmaxf(m1, __uint_as_float(r[e + 1]));
    m2 = fmaxf(m2, __uint_as_float(r[e + 2]));
    m3 = fmaxf(m3, __uint_as_float(r[e + 3]));
  }
  return fmaxf(fmaxf(m0, m1), fmaxf(m2, m3));
}


template <bool kVotes>
__global__ void __launch_bounds__(kThreads, 1)
score_tc_kernel(const __grid_constant__ CUtensorMap q_map, const __grid_constant__ CUtensorMap k_map,
                const ScoreArgs a) {
  constexpr int TILE_KEYS = kVotes ? 128 : 256;
  constexpr uint32_t STAGE_BYTES = TILE_KEYS * 256;
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long bars[18];
  __shared__ uint32_t tmem_slot;
  __shared__ Ctl ctl;
  // votes: -lse2 of the columns this warp reads, one copy per warp
  __shared__ __align__(16) float nlse2_s[kVotes ? kGroups * 4 : 1][kVotes ? 128 : 4];
  __shared__ float lse_s[kVotes ? 2 : 1][kVotes ? kMaxRows : 1];   // combined here: the LSE of the CTA's (at most two) units

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int cta = blockIdx.x;
  const int g_begin = cta * a.tiles_per_cta;
  const int g_end = min(a.total_tiles, g_begin + a.tiles_per_cta);
  const int nt = g_end - g_begin;
  const int Hkv = a.Hq / a.G;
  // The statistics walk their range upwards and the votes downwards: the keys that the pass ahead read last are still in
  // L2, and so are those that the votes read last when the calibration, upwards again, starts.
  // (the position inside the tile space is tracked incrementally: no division per tile)
  const int g_first = kVotes ? max(g_end - 1, g_begin) : g_begin;
  const int vu_begin = g_first / a.n_tiles, tile_begin = g_first - vu_begin * a.n_tiles;
  constexpr int kDir = kVotes ? -1 : 1;
  const int unit_tile0 = kVotes ? a.n_tiles - 1 : 0, past_tile = kVotes ? -1 : a.n_tiles;  // a virtual unit's first tile, past its last

  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t q_half_bytes = (uint32_t)a.block_rows * kLineBytes;
  const uint32_t q_blk_bytes = 2u * q_half_bytes;
  const uint32_t q_base = smem_base;
  const uint32_t k_base = q_base + (uint32_t)a.n_blocks * q_blk_bytes;

  const uint32_t bar0 = smem_u32(bars);
  const uint32_t q_full = bar0, q_empty = bar0 + 8u;
  auto full_k = [&](int s) { return bar0 + 8u * (2 + s); };
  auto empty_k = [&](int s) { return bar0 + 8u * (6 + s); };
  auto t_full = [&](int b) { return bar0 + 8u * (10 + b); };
  auto t_empty = [&](int b) { return bar0 + 8u * (14 + b); };

  if (tid == 0) {
    ctl.abort = 0;
    ctl.status = a.status;
    mbar_init(q_full, 1);
    mbar_init(q_empty, 1);
    for (int s = 0; s < 4; ++s) { mbar_init(full_k(s), 1); mbar_init(empty_k(s), 1); }
    for (int b = 0; b < kMaxBufs; ++b) {
      mbar_init(t_full(b), 1);
      mbar_init(t_empty(b), a.lg_bufs == 2 ? 128 : 256);   // a buffer is drained by one group or by a pair of them
    }
    fence_mbar_init();
  }
  if (warp == kMmaWarp) {
    tmem_alloc(smem_u32(&tmem_slot), kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = tmem_slot;
  pdl_wait();   // everything above ran beside the previous kernel's end; global memory from here on
  // (an error code is stored seconds into a wait, long after this; a memset ahead of the kernel would cost the chain
  // of programmatic launches 2 us)
  if (a.clear_status && blockIdx.x == 0 && tid == 0) *a.status = 0u;

  if (warp == kProducerWarp) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      tma_prefetch_desc(&q_map);
      tma_prefetch_desc(&k_map);
      int cur_vu = -1, seg = 0, vu = vu_begin, tile = tile_begin, unit = vu_begin / a.vu_per_unit;
      for (int i = 0; i < nt; ++i, tile += kDir) {
        if (tile == past_tile) { tile = unit_tile0; vu += kDir; unit = vu / a.vu_per_unit; }
        if (vu != cur_vu) {
          // the query rows of the next virtual unit replace the current ones once its MMAs are done
          if (seg > 0 && !mbar_wait(&ctl, q_empty, (seg - 1) & 1, (kVotes ? 36u : 16u) | ((unsigned)i << 8))) break;
          const int row0 = (vu - unit * a.vu_per_unit) * a.vu_rows;
          mbar_arrive_expect_tx(q_full, (uint32_t)a.n_blocks * q_blk_bytes);
          for (int blk = 0; blk < a.n_blocks; ++blk)
            for (int half = 0; half < 2; ++half)
              tma_load_3d(q_base + blk * q_blk_bytes + half * q_half_bytes, &q_map, q_full, half * kHalfCols,
                          row0 + blk * a.block_rows, unit);
          cur_vu = vu;
          ++seg;
        }
        const int s = i % a.stages;
        if (!mbar_wait(&ctl, empty_k(s), ((i / a.stages) & 1) ^ 1, (kVotes ? 31u : 11u) | ((unsigned)i << 8))) break;
        mbar_arrive_expect_tx(full_k(s), STAGE_BYTES);
        for (int half = 0; half < 2; ++half)
          tma_load_3d(k_base + s * STAGE_BYTES + half * (STAGE_BYTES / 2), &k_map, full_k(s), half * kHalfCols,
                      tile * TILE_KEYS, unit);
      }
    }
  } else if (__shfl_sync(0xffffffffu, warp, 0) == kMmaWarp) {
    // ------------------------------------------------------------ MMA issuer
    // The whole warp walks the loop and one lane issues: the values are then warp-uniform, and the operands
    // of an MMA come from uniform registers as they are.  With one lane in a loop of its own the eight MMAs of a job
    // took 560 cycles to issue and a job 1700 in all, which was the pace of the votes of 128 rows (64 units x 16384
    // keys: 64.8 -> 50 us, 5.3 TB/s of keys).  The shuffle makes the role of this warp uniform to the compiler; the
    // consumers keep the plain index, with which they need fewer registers.
    const uint32_t idesc = umma_idesc(128, kVotes ? a.block_rows : TILE_KEYS, false, false);
    // Descriptors are built once per buffer; a k-step adds a constant to the address field.
    const uint64_t dq0 = smem_desc_sw128(q_base, 16u, 1024u);
    const uint64_t dk0 = smem_desc_sw128(k_base, 16u, 1024u);
    const bool leader = elect_one();
    int seg = 0, j = 0, s = 0, tile = tile_begin;
    uint32_t s_ph = 0;
    bool first = true, ok = true;
    for (int i = 0; i < nt && ok; ++i) {
      if (first) {
        ok = __all_sync(0xffffffffu, mbar_wait_far(&ctl, q_full, seg & 1, (kVotes ? 32u : 12u) | ((unsigned)i << 8)));
        if (!ok) break;
        ++seg;
      }
      ok = __all_sync(0xffffffffu, mbar_wait_far(&ctl, full_k(s), s_ph, (kVotes ? 33u : 13u) | ((unsigned)i << 8)));
      if (!ok) break;
      const uint64_t kd = desc_advance(dk0, (uint32_t)s * STAGE_BYTES);
      for (int blk = 0; blk < a.n_blocks; ++blk, ++j) {
        const int buf = j & ((1 << a.lg_bufs) - 1);
        ok = __all_sync(0xffffffffu, mbar_wait_far(&ctl, t_empty(buf), ((j >> a.lg_bufs) & 1) ^ 1, (kVotes ? 34u : 14u) | ((unsigned)j << 8)));
        if (!ok) break;
        tc_fence_after_sync();
        const uint32_t d = tmem_base + (uint32_t)(buf << (9 - a.lg_bufs));
        const uint64_t qd = desc_advance(dq0, (uint32_t)blk * q_blk_bytes);
        // the second halves (k-steps 4..7) start half a tile further on
        const uint64_t kd2 = desc_advance(kd, STAGE_BYTES / 2), qd2 = desc_advance(qd, q_half_bytes);
        if (leader) {
          umma_ss_imm<0>(d, kVotes ? kd : qd, kVotes ? qd : kd, idesc);
#pragma unroll
          for (int kk = 1; kk < 4; ++kk)
            umma_ss_imm<1>(d, desc_advance(kVotes ? kd : qd, kk * 32u), desc_advance(kVotes ? qd : kd, kk * 32u), idesc);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            umma_ss_imm<1>(d, desc_advance(kVotes ? kd2 : qd2, kk * 32u), desc_advance(kVotes ? qd2 : kd2, kk * 32u), idesc);
          umma_commit(t_full(buf));
        }
        __syncwarp();
      }
      if (!ok) break;
      tile += kDir;
      first = tile == past_tile;
      if (first) tile = unit_tile0;
      if (leader) {
        umma_commit(empty_k(s));
        if (first || i == nt - 1) umma_commit(q_empty);
      }
      __syncwarp();
      if (++s == a.stages) { s = 0; s_ph ^= 1u; }
    }
  } else {
    // ------------------------------------------------------------ accumulator consumers
    // Thread ct of warpgroup grp owns TMEM lane ct.  The four groups form two pairs; the jobs (key
    // tile, row block) alternate between the pairs: pair p drains accumulator buffer p, each of its two
    // groups half of the columns.  With two row blocks a pair therefore always has the same one, with one
    // every second tile.  Votes of at most 128 window rows have four accumulators instead, one per group:
    // a job is as long as with 256 rows, where half a job per group would double what lies between two
    // (64 units x 16384 keys: whole call 199 -> 193 us).  While one pair waits for the MMAs of its next job (which cannot start before
    // the last columns of the current one have been read), the other, two warps per scheduler, keeps
    // the exponentials going; one warp per scheduler alone reaches less than half of their rate.
    // (Measured at 32 units x 32768 keys, votes: two groups on the same job 110 us, the groups stalling
    // together at every job boundary; two groups on alternate jobs 100 us; four accumulators of 128
    // columns 110 us, the narrower MMAs costing more than the wait they hide.)
    // What is left between two jobs is kept to a handful of instructions: everything that depends on
    // the virtual unit is worked out per segment (a run of tiles of one virtual unit), a job's own state
    // is a tile base and a phase bit, and the halves of a vote go out as they are, to be added by the
    // selection.  A warp's dependent scalar instructions cost some five cycles each: with a loop over
    // tiles and blocks, the running statistics in shared memory and the halves of a vote meeting there,
    // a job carried 190 instructions besides its exponentials, 800 cycles of about 5500.
    const int grp = warp >> 2, ct = tid & 127;
    const int pair = grp >> 1, half = grp & 1;
    const bool alone = kVotes && a.lg_bufs == 2;   // a buffer per group
    const int blk = a.n_blocks > 1 ? pair : 0, step = a.n_blocks > 1 ? 1 : (alone ? 4 : 2);
    const int buf = alone ? grp : pair;
    // this group's columns of the buffer: [col0, col0 + cw), cw 64, 96 or 128
    const int cw = kVotes ? (alone ? a.block_rows : a.block_rows >> 1) : TILE_KEYS / 2, col0 = alone ? 0 : half * cw;
    const uint32_t taddr = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((buf << (9 - a.lg_bufs)) + col0);
    const uint32_t bar_full = t_full(buf), bar_empty = t_empty(buf);
    const f32x2 sc = pack2(a.scale2);
    uint32_t ph = 0;
    bool ok = true;

    const int unit_lo = g_begin / a.n_tiles;
    const bool combine = kVotes && a.stats.part != nullptr;
    if (combine) {
      // Row LSE of this CTA's units from the partial statistics, by the consumers while the first keys are on their way:
      // cheaper than a kernel of its own as long as the partials are few (see votes_combine_stats).
      const int tpr = 1 << a.lg_tpr, row = tid >> a.lg_tpr, sub = tid & (tpr - 1);
      const int unit_hi = (g_end - 1) / a.n_tiles;
      for (int unit = unit_lo; unit <= unit_hi; ++unit) {
        float m = -1e30f, l = 0.f;
        if (row < a.GW) {
          int n;
          const float2* p = a.stats.of(unit, a.GW, row, &n);
          for (int i0 = sub; i0 < n; i0 += 4 * tpr) {
            float2 v[4];
            float mn = m;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              v[k] = i0 + k * tpr < n ? __ldcg(p + i0 + k * tpr) : make_float2(-1e30f, 0.f);
              mn = fmaxf(mn, v[k].x);
            }
            l *= exp2_unbiased(m - mn);
#pragma unroll
            for (int k = 0; k < 4; ++k) l += v[k].y * exp2_unbiased(v[k].x - mn);
            m = mn;
          }
        }
        // (the maximum first, then one factor per thread: factors on every level of the exchange would add up their errors)
        float M = m;
        for (int o = 1; o < tpr; o <<= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
        l *= exp2_unbiased(m - M);
        for (int o = 1; o < tpr; o <<= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (row < a.GW && sub == 0) {
          const float lse = (M + log2f(l)) * kLn2;
          lse_s[unit - unit_lo][row] = lse;
          const int tile0 = unit * a.n_tiles;   // the CTA that has the unit's first tile hands it on
          if (g_begin <= tile0 && tile0 < g_end) a.lse_out[(size_t)unit * a.GW + row] = lse;
        }
      }
      asm volatile("barrier.cta.sync 1, %0;" ::"n"(kGroups * 128) : "memory");
    }
    int seg0 = 0, seg_tile0 = tile_begin, vu = vu_begin;
    while (seg0 < nt && ok) {
      const int seg_n = min(nt - seg0, kVotes ? seg_tile0 + 1 : a.n_tiles - seg_tile0);
      const int unit = vu / a.vu_per_unit, row0 = (vu - unit * a.vu_per_unit) * a.vu_rows;
      const int hq0 = (unit / Hkv) * a.Hq + (unit % Hkv) * a.G;
      float* vote_out = nullptr;                 // votes: this group's part of the unit's votes
      float2 ml = make_float2(-1e30f, 0.f);      // statistics: running (max, sum) of this thread's row
      int lim = 0;                               // statistics: the last key the row may see (causal in the window)
      if (kVotes) {
        // this warp's copy of -lse2 of its columns' window rows (-inf for the padding rows); a copy per
        // warp, so that no barrier wider than a warp is needed here
        __syncwarp();
        for (int c = lane; c < cw; c += 32) {
          const int r = blk * a.block_rows + col0 + c;
          const float lse = r >= a.GW ? INFINITY : combine ? lse_s[unit - unit_lo][r] : a.row_lse[(size_t)hq0 * a.W + r];
          nlse2_s[warp][c] = -lse * kLog2e;
        }
        __syncwarp();
        const int part = alone ? 0 : 2 * blk + half, units = a.total_tiles / a.n_tiles;
        vote_out = a.vote_parts + ((size_t)part * units + unit) * a.n_cand;
      } else {
        lim = min(a.L - 1, a.n_cand + (row0 + blk * 128 + ct) % a.W);
      }
      // the first tile of the segment that is this buffer's: tile i of the CTA goes to buffer i % step
      const int first = (buf - seg0) & (step - 1);
      int key0 = (seg_tile0 + kDir * first) * TILE_KEYS;
#pragma unroll 1
      for (int i = first; i < seg_n; i += step, key0 += kDir * step * TILE_KEYS) {
        ok = mbar_wait(&ctl, bar_full, ph, (kVotes ? 35u : 15u) | ((unsigned)i << 8));
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        ph ^= 1u;
        tc_fence_after_sync();
        uint32_t ra[32], rb[32];
        if (kVotes) {
          f32x2 acc0 = 0ull, acc1 = 0ull;  // the vote of this thread's key over this group's columns
          auto add32 = [&](const uint32_t (&r)[32], int c0) {
            const float* nl = nlse2_s[warp] + c0;
#pragma unroll
            for (int e = 0; e < 32; e += 4) {
              const ulonglong2 n4 = *reinterpret_cast<const ulonglong2*>(nl + e);
              const f32x2 x0 = fma2(pack2(r[e], r[e + 1]), sc, n4.x), x1 = fma2(pack2(r[e + 2], r[e + 3]), sc, n4.y);
              acc0 = add_exp2_pair<true>(acc0, x0, e / 2);
              acc1 = add_exp2_pair<true>(acc1, x1, e / 2 + 1);
            }
          };
          // chunks of 32 columns alternate between the two register sets; unrolled, since a loop with the
          // conditions inside took 163 instead of 134 thousand cycles
          auto drain = [&](auto cw_tag) __attribute__((always_inline)) {
            constexpr int kCw = decltype(cw_tag)::value;
            tmem_ld32_issue(taddr, ra);
#pragma unroll
            for (int c0 = 0; c0 < kCw; c0 += 64) {
              tmem_ld_wait(ra);
              if (c0 + 32 < kCw) tmem_ld32_issue(taddr + c0 + 32, rb);
              else { tc_fence_before_sync(); mbar_arrive(bar_empty); }   // all of it is in registers
              add32(ra, c0);
              if (c0 + 32 < kCw) {
                tmem_ld_wait(rb);
                if (c0 + 64 < kCw) tmem_ld32_issue(taddr + c0 + 64, ra);
                else { tc_fence_before_sync(); mbar_arrive(bar_empty); }
                add32(rb, c0 + 32);
              }
            }
          };
          if (cw == 128) drain(std::integral_constant<int, 128>{});
          else if (cw == 64) drain(std::integral_constant<int, 64>{});
          else drain(std::integral_constant<int, 96>{});
          const float2 acc = unpack2(add2(acc0, acc1));
          if (key0 + ct < a.n_cand) vote_out[key0 + ct] = acc.x + acc.y;
        } else {
          const int l0 = lim - (key0 + half * cw);   // index of the row's last key among this group's keys of the tile
          const bool full = __all_sync(0xffffffffu, l0 >= cw - 1);
          auto fold32 = [&](uint32_t (&r)[32], int c0) {
            if (!full) {
#pragma unroll
              for (int e = 0; e < 32; ++e)
                if (c0 + e > l0) r[e] = 0xff800000u;  // -inf
            }
            const float m_new = fmaxf(ml.x, max_32(r) * a.scale2);
            ml.y = fmaf(ml.y, ex2_approx(ml.x - m_new), sum_exp2_32(r, sc, pack2(-m_new)));
            ml.x = m_new;
          };
          tmem_ld32_issue(taddr, ra);
#pragma unroll
          for (int c0 = 0; c0 < TILE_KEYS / 2; c0 += 64) {
            tmem_ld_wait(ra);
            tmem_ld32_issue(taddr + c0 + 32, rb);
            fold32(ra, c0);
            tmem_ld_wait(rb);
            if (c0 + 64 < TILE_KEYS / 2) {
              tmem_ld32_issue(taddr + c0 + 64, ra);
            } else {
              tc_fence_before_sync();
              mbar_arrive(bar_empty);  // the accumulator is in registers: hand the buffer back early
            }
            fold32(rb, c0 + 32);
          }
        }
      }
      if (!kVotes && ok) {
        // this group's partial (max, sum) of its row; with one row block both pairs have one
        const int slot = cta - (vu * a.n_tiles) / a.tiles_per_cta;
        const int row = row0 + blk * 128 + ct, n_part = a.n_blocks > 1 ? 2 : 4;
        if (row < a.GW)
          a.stat_part[(((size_t)hq0 * a.W + row) * a.max_slots + slot) * n_part + (a.n_blocks > 1 ? half : grp)] = ml;
      }
      seg0 += seg_n;
      seg_tile0 = unit_tile0;
      vu += kDir;
    }
  }

  // ---------------------------------------------------------------- teardown (every path)
  if (ctl.abort) {
    for (int i = 0; i < 50; ++i) __nanosleep(20000);  // let TMA copies still in flight land
  }
  tc_fence_before_sync();
  __syncthreads();
  // Every warp of the CTA is done: the next kernel's CTAs may set themselves up while this one winds
  // down.  (A trigger that any thread reaches earlier counts for the whole CTA: with the idle lanes of
  // the producer and issuing warps passing it at the kernel's top, the successors' CTAs sat beside
  // the running ones for the kernel's whole length and the compress step was 12 % slower.)
  pdl_trigger();
  if (warp == kMmaWarp) tmem_dealloc(tmem_base, kTmemCols);
}

// Combine the partial statistics of every observation row into its natural-log LSE, a warp per row (a thread
// per row walked up to a hundred partials one load after the other: 18.6 us for one prompt of 131072 keys).
__global__ void __launch_bounds__(256)
row_lse_from_parts_kernel(const StatParts stats, float* __restrict__ row_lse, int rows, int GW) {
  pdl_trigger();
  pdl_wait();
  const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= rows) return;
  const int unit = r / GW;
  int n;
  const float2* p = stats.of(unit, GW, r - unit * GW, &n);
  float m = -INFINITY, l = 0.f;
  for (int i = lane; i < n; i += 32) {
    const float2 q = p[i];
    const float mn = fmaxf(m, q.x);
    l = l * exp2_unbiased(m - mn) + q.y * exp2_unbiased(q.x - mn);
    m = mn;
  }
  const float M = warp_max(m);
  l = warp_sum(m > -INFINITY ? l * exp2_unbiased(m - M) : 0.f);
  if (lane == 0) row_lse[r] = (M + log2f(l)) * kLn2;
}

__global__ void add_votes_kernel(float* __restrict__ vote, const float* __restrict__ parts, int n_parts, size_t n) {
  pdl_trigger();
  pdl_wait();
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float x = parts[i];
  for (int p = 1; p < n_parts; ++p) x += parts[(size_t)p * n + i];
  vote[i] = x;
}

// The query rows of a virtual unit and the ring of key tiles share this much, however they divide it.
constexpr int kSmemMax = 192 * 1024 + 1024;

template <bool kVotes>
cudaError_t launch_score(const CUtensorMap& qm, const CUtensorMap& km, const ScoreArgs& a, int smem, cudaStream_t st) {
  static OncePerDevice granted;
  if (smem > kSmemMax) return cudaErrorInvalidValue;
  cudaError_t e = grant_smem(score_tc_kernel<kVotes>, kSmemMax, granted);
  if (e != cudaSuccess) return e;
  const int grid = (a.total_tiles + a.tiles_per_cta - 1) / a.tiles_per_cta;
  return launch_pdl(score_tc_kernel<kVotes>, dim3(grid), dim3(kThreads), (size_t)smem, st, qm, km, a);
}

// Equal contiguous tile ranges over at most one CTA per SM.
void partition_tiles(ScoreArgs& a, int virtual_units) {
  a.total_tiles = virtual_units * a.n_tiles;
  const int ctas = a.total_tiles < kSms ? a.total_tiles : kSms;
  a.tiles_per_cta = (a.total_tiles + ctas - 1) / ctas;
}

}  // namespace

// Number of key-range splits per work group so that `groups * splits` CTAs fill whole waves of
// the 148 SMs (one CTA per SM) while every CTA keeps at least `min_tiles` tiles.
int pick_tile_splits(int groups, int n_tiles, int min_tiles) {
  int max_s = n_tiles / (min_tiles > 0 ? min_tiles : 1);
  if (max_s < 1) max_s = 1;
  if (max_s > 64) max_s = 64;
  int best = 1;
  double best_eff = 0.0;
  for (int s = 1; s <= max_s; ++s) {
    const long long ctas = (long long)groups * s;
    const long long waves = (ctas + kSms - 1) / kSms;
    const double eff = (double)ctas / (double)(waves * kSms);
    if (eff > best_eff + 0.02) { best_eff = eff; best = s; }
  }
  return best;
}

bool score_tc_supported(const CompressGeom& g) {
  return !g.keep_all && g.G * g.W <= kMaxRows && g.W <= 128 && g.n_cand >= 1;
}

namespace {

// The statistics' tile partition, which the kernels that combine its partials need too.
void plan_stats(const CompressGeom& g, ScoreArgs& a) {
  const int GW = g.G * g.W;
  a.Hq = g.Hq; a.G = g.G; a.W = g.W; a.L = g.L; a.n_cand = g.n_cand; a.GW = GW;
  a.vu_per_unit = (GW + 255) / 256;
  a.vu_rows = 256;
  a.n_blocks = GW <= 128 ? 1 : 2;
  a.block_rows = 128;
  a.n_tiles = (g.L + 255) / 256;
  partition_tiles(a, g.units * a.vu_per_unit);
  a.max_slots = (a.n_tiles + a.tiles_per_cta - 1) / a.tiles_per_cta + 1;
}

StatParts stat_parts(const ScoreArgs& a, const float2* part) {
  return StatParts{part, a.vu_per_unit, a.n_tiles, a.tiles_per_cta, a.max_slots, a.n_blocks > 1 ? 2 : 4};
}

void plan_votes(const CompressGeom& g, ScoreArgs& a) {
  const int GW = g.G * g.W;
  a.Hq = g.Hq; a.G = g.G; a.W = g.W; a.L = g.L; a.n_cand = g.n_cand; a.GW = GW;
  a.vu_per_unit = 1;
  a.vu_rows = 0;
  // One accumulator of up to 256 row columns per (key tile, row block).
  a.n_blocks = (GW + 255) / 256;
  a.block_rows = ((GW + a.n_blocks - 1) / a.n_blocks + 63) / 64 * 64;
  a.lg_bufs = a.block_rows <= 128 ? 2 : 1;
  a.n_tiles = (g.n_cand + kTileKeys - 1) / kTileKeys;
  partition_tiles(a, g.units);
}

}  // namespace

size_t row_stats_tc_slots(const CompressGeom& g) {
  ScoreArgs a{};
  plan_stats(g, a);
  return (size_t)a.max_slots * stat_parts(a, nullptr).n_part;
}

// Whether the votes combine the partial statistics themselves: every CTA then reads the partials of its one or two
// units, so they must be few.  Whole compress calls with the kernel of its own and without: 8 units of 9 KB 28.2 -> 27.6 us,
// 32 of 24 KB (32768 keys) about 1 % less, 8 of 69 KB (8192 keys) 44.6 -> 45.2.
bool votes_combine_stats(const CompressGeom& g) {
  ScoreArgs st{}, vt{};
  plan_stats(g, st);
  plan_votes(g, vt);
  const StatParts p = stat_parts(st, nullptr);
  return vt.tiles_per_cta <= vt.n_tiles && (size_t)st.GW * p.max_slots * p.n_part * sizeof(float2) <= 32768;
}

// Statistics of the G*W observation rows of every unit: the partials and, unless the votes combine them, the row LSE
// into ws.row_lse.  `first`: of a call, the kernel then clears the workspace's error word.
cudaError_t launch_row_stats_tc(const CompressGeom& g, const CompressWs& ws, const void* Q_obs, const void* K,
                                char* wsp, bool first, bool combine, cudaStream_t st) {
  const int GW = g.G * g.W;
  ScoreArgs a{};
  a.clear_status = first;
  plan_stats(g, a);
  a.stages = 2;  // 64 KB tiles of 256 keys
  a.lg_bufs = 1;
  a.scale2 = g.scale2;
  a.stat_part = (float2*)(wsp + ws.stat_part);
  a.status = (unsigned*)(wsp + ws.status);
  CUtensorMap qm, km;
  const uint64_t qd[2] = {(uint64_t)GW, (uint64_t)g.units}, qs[2] = {256, (uint64_t)GW * 256};
  const uint32_t qb[2] = {128, 1};
  const uint64_t kd[2] = {(uint64_t)g.L, (uint64_t)g.units}, ks[2] = {256, (uint64_t)g.L * 256};
  const uint32_t kb[2] = {256, 1};
  if (!make_tensor_map_bf16(&qm, Q_obs, 3, qd, qs, qb) || !make_tensor_map_bf16(&km, K, 3, kd, ks, kb))
    return cudaErrorInvalidValue;
  const int smem = a.n_blocks * 128 * 256 + a.stages * 256 * 256 + 1024;
  cudaError_t e = launch_score<false>(qm, km, a, smem, st);
  if (e != cudaSuccess) return e;
  count_launch(1);
  if (combine) {
    const int rows = g.B * g.Hq * g.W;
    e = launch_pdl(row_lse_from_parts_kernel, dim3((rows + 7) / 8), dim3(256), 0, st, stat_parts(a, a.stat_part),
                   (float*)(wsp + ws.row_lse), rows, GW);
    count_launch(1);
  }
  return e != cudaSuccess ? e : cudaGetLastError();
}

// Parts of a candidate's vote that launch_votes_tc leaves: one per row block and column half, one in all for
// at most 128 rows.
int votes_tc_parts(const CompressGeom& g) { return g.G * g.W <= 128 ? 1 : 2 * ((g.G * g.W + 255) / 256); }

// Partial votes of every candidate key, into ws.vote_parts; the selection adds them up.  row_lse null: combined from the
// partials that the statistics left in the workspace, and written to ws.row_lse.
cudaError_t launch_votes_tc(const CompressGeom& g, const CompressWs& ws, const void* Q_obs, const void* K,
                            const float* row_lse, char* wsp, bool first, cudaStream_t st) {
  const int GW = g.G * g.W;
  ScoreArgs a{};
  a.clear_status = first;
  plan_votes(g, a);
  if (!row_lse) {
    ScoreArgs sa{};
    plan_stats(g, sa);
    a.stats = stat_parts(sa, (const float2*)(wsp + ws.stat_part));
    a.lse_out = (float*)(wsp + ws.row_lse);
    while (a.lg_tpr < 5 && (GW << (a.lg_tpr + 1)) <= kGroups * 128) ++a.lg_tpr;
  }
  const int q_bytes = a.n_blocks * a.block_rows * 256;
  a.stages = q_bytes <= 65536 ? 4 : (q_bytes <= 98304 ? 3 : 2);
  a.scale2 = g.scale2;
  a.row_lse = row_lse;
  a.vote_parts = (float*)(wsp + ws.vote_parts);
  a.status = (unsigned*)(wsp + ws.status);
  CUtensorMap qm, km;
  const uint64_t qd[2] = {(uint64_t)GW, (uint64_t)g.units}, qs[2] = {256, (uint64_t)GW * 256};
  const uint32_t qb[2] = {(uint32_t)a.block_rows, 1};
  const uint64_t kd[2] = {(uint64_t)g.L, (uint64_t)g.units}, ks[2] = {256, (uint64_t)g.L * 256};
  const uint32_t kb[2] = {(uint32_t)kTileKeys, 1};
  if (!make_tensor_map_bf16(&qm, Q_obs, 3, qd, qs, qb) || !make_tensor_map_bf16(&km, K, 3, kd, ks, kb))
    return cudaErrorInvalidValue;
  const int smem = q_bytes + a.stages * kKvTileBytes + 1024;
  cudaError_t e = launch_score<true>(qm, km, a, smem, st);
  if (e != cudaSuccess) return e;
  count_launch(1);
  return cudaGetLastError();
}

// The parts added into ws.vote, for the selection that does not add them itself.
cudaError_t launch_add_votes(const CompressGeom& g, const CompressWs& ws, char* wsp, cudaStream_t st) {
  const size_t n = (size_t)g.units * g.n_cand;
  cudaError_t e = launch_pdl(add_votes_kernel, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, st, (float*)(wsp + ws.vote),
                             (const float*)(wsp + ws.vote_parts), votes_tc_parts(g), n);
  if (e != cudaSuccess) return e;
  count_launch(1);
  return cudaGetLastError();
}

}  // namespace calidrop
