// The whole compress-and-calibrate step of a (batch, kv head) unit in one kernel, for the calls whose units are small
// enough that a cluster of CTAs can walk one: statistics, votes, pooled top-k, calibration and compaction without a
// launch, a pass over global memory or an idle GPU between them.
//
// A cluster of 1..16 CTAs shares a unit; CTA r owns the key tiles [r * T, (r + 1) * T) of 128 keys.  Phases:
//   S  row statistics: S = Q K^T with the window rows on the tensor-memory lanes, (max, sum) per row, combined over the
//      cluster into the row LSE (left out when the caller supplies it)
//   V  votes: S^T = K Q^T with the keys on the lanes, the vote of a key is a per-thread sum over the rows
//   select: pooling and an exact radix select over the cluster; the votes never leave the CTA but for the outputs
//   (for a caller's kept list, calidrop_calibrate, V and the selection fall away)
//   C  calibration: S = Q_c K^T again, probabilities of the evicted keys as the A operand of O += P V
//   reduce: every CTA finishes a share of the calibration rows from the partial O that all left in the workspace; one warp copies the
//      retained rows meanwhile (up to kCopyRows a CTA: more of them take a kernel on all SMs behind this one)
// K is streamed once per phase through one TMA ring (from L2 after the first time), so the keys of a CTA are not limited
// by its shared memory, and the loads of phase C run during the selection.  What the CTAs of a cluster tell each
// other is PUSHED with asynchronous stores that report their bytes to an mbarrier of the receiver; only the partial O, which is
// larger, goes through the workspace.
// Warp roles: sixteen consumer warps in four groups (each a quarter of a tile's columns, so that all of them share every
// tile), a TMA producer, an MMA issuer for S and S^T, one for P.V, a warp that compacts the retained rows.
//
// What bounds it: the latency of a chain of some fifteen steps (clock stamps, 8 units x 2048 keys x 32 rows, thousand cycles
// of 30: start 2, S 3.5, row LSE 3.3, V 1.8, staging 1.6, select 8.5, C 2.3, O 2, exchange and end 5); for longer units
// the exponentials, one per logit and phase (see exp2.cuh), and the warps' issue slots beside them: 1250 cycles a tile and
// phase for 1024 exponential-unit cycles, whatever share of them is on the FMA pipe.  The code is kept small on purpose
// (loops not unrolled, waits out of line): most of it runs once per launch, and 260 KB of it took 20 us
// where 110 KB take 16.6.  Five to six kernels -> this one, us: 8 units x 2048 keys x 32 rows 28.3 -> 16.7, 8 x 8192 x 128 45.0 ->
// 32.2, 16 x 5003 x 120 with the caller's row LSE and a calibration size 42.8 -> 28.5.
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "exp2.cuh"
#include "internal.h"
#include "tc_common.cuh"

namespace calidrop {

namespace {

using namespace tc;

constexpr int kGroups = 4;
constexpr int kConsumers = kGroups * 128;
constexpr int kProducerWarp = kGroups * 4;
constexpr int kMmaWarp = kProducerWarp + 1;
constexpr int kPvWarp = kProducerWarp + 2;
constexpr int kGatherWarp = kProducerWarp + 3;
constexpr int kThreads = kGatherWarp * 32 + 32;   // twenty warps: with one more, a thread would have 80 registers, not 96
constexpr int kMaxRows = 128;              // G * W of a unit
constexpr int kMaxClu = 16;
constexpr int kMaxTiles = 64;              // tiles of a CTA: the counts of a histogram are 16 bits wide
constexpr int kMinStages = 4, kMaxStages = 6;
constexpr int kBars = 46;
constexpr int kHaloMax = 64;               // widest half pool
constexpr int kAccBufs = 4;                // phases S and V: accumulators of 128 columns
constexpr int kCalBufs = 3;                // phase C: S/P buffers of 128 columns, O behind them
constexpr uint32_t kColO = kCalBufs * 128;
constexpr int kTileBytes = kKvTileBytes;   // 32 KB
constexpr int kOStride = kD + 4;           // row stride of the partial O in shared memory: no bank conflicts
constexpr int kQuarterTiles = 16;          // up to this many tiles the four groups share a tile's votes
constexpr int kHistCopies = 8;
// Retained rows of a CTA that this kernel compacts itself.  Beyond, the SMs without a CTA of it are missed, and a kernel of their own
// behind it compacts the rows, us: 100 units x 4000 keys, 3200 of them kept, 159 -> 133; 8 x 30000, 24000 kept, 113 -> 91; 1 x
// 30000, 12000 kept, 51 -> 46; 40 x 8000, 1600 kept (533 a CTA) 71.6 and 72.2; 8 x 8192, 1638 kept (164 a CTA) 29.5 and 30.9.
constexpr int kCopyRows = 512;
constexpr int kSmemMax = 221 * 1024;       // dynamic; the static arrays take less than 6 KB

struct ClusterArgs {
  int Hq, G, W, L, n_cand, n_cal, GW, cal_rows;
  int n_tiles, tiles_per_cta, n_clu, stages;
  int lg_rep, lg_rep_c;   // copies of the window rows / calibration rows on the 128 lanes
  int n_pad;              // phase V: columns of an accumulator, 32, 64 or 128
  int pool, k_sel, n_kept, n_calib, bitmap_words;
  int n_copy;             // retained rows that this kernel compacts: all of them or none
  int stage_off, keys_off, mask_off;   // bytes from the scratch area's start
  float scale2;
  const float* row_lse;   // the caller's, or null
  float* row_lse_out;
  float* vote;
  float* pooled;
  uint32_t* mask2;        // kSized: bit set = not one of the calibrated evicted rows
  int32_t* kept_idx;
  const __nv_bfloat16* Q_obs;
  float* O_c;
  float* LSE_c;
  __nv_bfloat16* C_q;
  float* o_part;          // [unit][cluster rank][cal_rows][128]: partial O of the CTAs
  float* l_part;          // ... and their row sums
  GatherArgs gather;
  unsigned* status;
};

// ---------------------------------------------------------------- cluster helpers
__device__ __forceinline__ uint32_t peer_addr(uint32_t local, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
  return r;
}
__device__ __forceinline__ void push_u32(uint32_t remote, uint32_t x, uint32_t remote_bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.u32 [%0], %1, [%2];" ::"r"(remote), "r"(x),
               "r"(remote_bar)
               : "memory");
}
__device__ __forceinline__ void push_f32x2(uint32_t remote, float x, float y, uint32_t remote_bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(remote),
               "f"(x), "f"(y), "r"(remote_bar)
               : "memory");
}
__device__ __forceinline__ void push_u32x4(uint32_t remote, uint4 v, uint32_t remote_bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.u32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(
                   remote),
               "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(remote_bar)
               : "memory");
}
__device__ __forceinline__ void arrive_peer(uint32_t remote_bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(remote_bar) : "memory");
}
// A bounded wait for what the peers of the cluster wrote ahead of their arrivals.
__device__ __forceinline__ bool mbar_wait_cluster(Ctl* ctl, uint32_t bar, uint32_t parity, unsigned code) {
  if (!mbar_wait_far(ctl, bar, parity, code)) return false;
  asm volatile("fence.acq_rel.cluster;" ::: "memory");
  return true;
}

__device__ __forceinline__ bool nonfinite_bf16x4(uint2 x) {
  return (x.x & 0x7f80u) == 0x7f80u || (x.x & 0x7f800000u) == 0x7f800000u || (x.y & 0x7f80u) == 0x7f80u ||
         (x.y & 0x7f800000u) == 0x7f800000u;
}
// Elements 4 lane .. 4 lane + 3 of a row's partial O over n keys, for a row with copies whose copies added up to NaN: a copy has
// zeros for the other copies' keys, and zero times an infinite value of V is NaN where the row itself has a probability above zero.
// Only products that are not finite decide such an element (`l`, the row's sum, tells whether a probability can be one); none
// found, it stays as it is.  A whole warp works on a row, four elements a lane, until all of its NaN are settled.  Out of line:
// finite inputs never get here, and the instruction fetch of code beside the loop costs all.  (Every lane for itself, with a
// product of 128 terms for each key that it met, a call of 8 units x 8192 keys x 64 calibration rows whose values were all infinite
// took 11.2 ms; a key per lane 1.5, bound by the uncoalesced loads; now 0.8, and 0.05 where both signs meet.)
__device__ __noinline__ float4 refold_nonfinite(float4 o, const __nv_bfloat16* q, const __nv_bfloat16* K, const __nv_bfloat16* V,
                                                int n, const uint32_t* mask, float scale2, float nlse2, float l, int lane) {
  constexpr int kKeys = 8;   // at a time
  if (isnan(l)) return o;
  const bool all = !isfinite(l);
  const uint2 q4 = reinterpret_cast<const uint2*>(q)[lane];
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
  for (int t0 = 0; t0 < n; t0 += kKeys) {
    uint2 v[kKeys], k[kKeys];
    bool any = false;
#pragma unroll
    for (int j = 0; j < kKeys; ++j) {
      const size_t at = (size_t)min(t0 + j, n - 1) * (kD / 4) + lane;
      v[j] = reinterpret_cast<const uint2*>(V)[at];
      k[j] = reinterpret_cast<const uint2*>(K)[at];
    }
#pragma unroll
    for (int j = 0; j < kKeys; ++j) any = any || nonfinite_bf16x4(v[j]);
    if (!__any_sync(0xffffffffu, all || any)) continue;
    float s[kKeys], mine = 0.f;   // mine: of key lane % kKeys
#pragma unroll
    for (int j = 0; j < kKeys; ++j) {
      s[j] = fmaf(bf16_hi(q4.x), bf16_hi(k[j].x), bf16_lo(q4.x) * bf16_lo(k[j].x));
      s[j] = fmaf(bf16_hi(q4.y), bf16_hi(k[j].y), fmaf(bf16_lo(q4.y), bf16_lo(k[j].y), s[j]));
    }
#pragma unroll
    for (int o2 = 16; o2 > 0; o2 >>= 1)
#pragma unroll
      for (int j = 0; j < kKeys; ++j) s[j] += __shfl_xor_sync(0xffffffffu, s[j], o2);
#pragma unroll
    for (int j = 0; j < kKeys; ++j) mine = lane % kKeys == j ? s[j] : mine;
    const int t = min(t0 + lane % kKeys, n - 1);
    const float p = (mask[t >> 5] >> (t & 31)) & 1u ? 0.f : __bfloat162float(__float2bfloat16(exp2f(fmaf(mine, scale2, nlse2))));
#pragma unroll
    for (int j = 0; j < kKeys; ++j) {
      const float pj = __shfl_sync(0xffffffffu, p, j);
      if (t0 + j < n && (all || nonfinite_bf16x4(v[j]))) {
        acc.x = fmaf(pj, bf16_lo(v[j].x), acc.x);
        acc.y = fmaf(pj, bf16_hi(v[j].x), acc.y);
        acc.z = fmaf(pj, bf16_lo(v[j].y), acc.z);
        acc.w = fmaf(pj, bf16_hi(v[j].y), acc.w);
      }
    }
    const bool settled = (isnan(acc.x) || !isnan(o.x)) && (isnan(acc.y) || !isnan(o.y)) && (isnan(acc.z) || !isnan(o.z)) &&
                         (isnan(acc.w) || !isnan(o.w));
    if (__all_sync(0xffffffffu, settled)) break;
  }
  return make_float4(isnan(o.x) && !isfinite(acc.x) ? acc.x : o.x, isnan(o.y) && !isfinite(acc.y) ? acc.y : o.y,
                     isnan(o.z) && !isfinite(acc.z) ? acc.z : o.z, isnan(o.w) && !isfinite(acc.w) ? acc.w : o.w);
}

// Columns of this thread's lane: the load, and its completion (see tmem_ld32_issue).
template <int N>
__device__ __forceinline__ void tmem_issue(uint32_t taddr, uint32_t (&r)[N]) {
  if constexpr (N == 32) {
    tmem_ld32_issue(taddr, r);
  } else if constexpr (N == 16) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
  } else {
    static_assert(N == 8, "8, 16 or 32 columns");
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
  }
}
template <int N>
__device__ __forceinline__ void tmem_wait(uint32_t (&r)[N]) {
  if constexpr (N == 32) {
    tmem_ld_wait(r);
  } else if constexpr (N == 16) {
    asm volatile("tcgen05.wait::ld.sync.aligned;\n"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
                 :
                 : "memory");
  } else {
    asm volatile("tcgen05.wait::ld.sync.aligned;\n"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])
                 :
                 : "memory");
  }
}
// kGiven: the kept list is the caller's; V and the selection fall away.
template <bool kSized, bool kGiven>
__global__ void __launch_bounds__(kThreads, 1)
compress_cluster_kernel(const __grid_constant__ CUtensorMap q_map, const __grid_constant__ CUtensorMap qc_map,
                        const __grid_constant__ CUtensorMap k_map, const __grid_constant__ CUtensorMap v_map,
                        const ClusterArgs a) {
  constexpr int kThr = kSized ? 2 : 1;
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long bars[kBars];
  __shared__ uint32_t tmem_slot;
  __shared__ Ctl ctl;
  __shared__ int next_row;                            // of this CTA's share of the kept list
  __shared__ __align__(16) float nlse2_s[kMaxRows];   // -row LSE in the log2 domain
  __shared__ float lse_s[kMaxRows];                   // row LSE, natural
  __shared__ float l_s[kGroups][128];                 // phase C: row sums of the groups
  __shared__ unsigned sel_bin[kThr], sel_k[kThr], sel_all[kThr];
  __shared__ unsigned wcnt[kThr][16][2];              // keys above / equal to a threshold, per warp
  __shared__ unsigned ccnt[kThr][kMaxClu][2];         // ... per CTA of the cluster

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = blockIdx.x, n_clu = a.n_clu, unit = blockIdx.y;   // (the grid's x extent is one cluster)
  const int Hkv = a.Hq / a.G;
  const int tile0 = rank * a.tiles_per_cta, c0 = tile0 * kTileKeys;
  const int nt = min(a.tiles_per_cta, a.n_tiles - tile0);            // at least one
  const int n_own = max(0, min(nt * kTileKeys, a.n_cand - c0));      // candidates of this CTA
  const int nC = (n_own + kTileKeys - 1) / kTileKeys, nV = kGiven ? 0 : nC, nS = a.row_lse ? 0 : nt;

  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  unsigned char* const smem_al = smem_raw + (smem_base - smem_u32(smem_raw));
  const uint32_t q_base = smem_base, ring = q_base + kTileBytes;
  float* const obuf = reinterpret_cast<float*>(smem_al + kTileBytes);   // the ring, once its last tile is consumed
  unsigned char* const scratch = smem_al + kTileBytes + a.stages * kTileBytes;
  // scratch, in turn: the statistics' exchange; partial votes; histograms
  float2* const xs = reinterpret_cast<float2*>(scratch);                          // [kGroups][128]
  float2* const lse_in = xs + kGroups * 128;                                      // [n_clu][128], pushed by the peers
  float* const vparts = reinterpret_cast<float*>(scratch);                        // [kGroups][nt * 128]
  unsigned* const hist = reinterpret_cast<unsigned*>(scratch);                    // [kThr][256][kHistCopies]
  unsigned short* const counts = reinterpret_cast<unsigned short*>(hist + kThr * 256 * kHistCopies);
  auto counts_of = [&](int buf, int x, int r) { return counts + ((buf * kThr + x) * n_clu + r) * 256; };
  float* const stage = reinterpret_cast<float*>(scratch + a.stage_off);           // votes with the pool's halo
  unsigned* const keys = reinterpret_cast<unsigned*>(scratch + a.keys_off);       // [tiles * 128], pooled votes
  uint32_t* const mask_s = reinterpret_cast<uint32_t*>(scratch + a.mask_off);     // [tiles][4], bit set = not calibrated

  const uint32_t bar0 = smem_u32(bars);
  const uint32_t q_full = bar0, q_empty = bar0 + 8u, o_full = bar0 + 16u;
  const uint32_t x_lse = bar0 + 24u, x_halo = bar0 + 32u, x_kept = bar0 + 40u, x_o = bar0 + 48u;
  auto x_hist = [&](int b) { return bar0 + 8u * (7 + b); };
  // (K and V tiles have barriers of their own: each issuer waits for every phase of its, and a parity never means another)
  auto full_k = [&](int s) { return bar0 + 8u * (9 + s); };
  auto full_v = [&](int s) { return bar0 + 8u * (40 + s); };
  auto empty = [&](int s) { return bar0 + 8u * (15 + s); };
  auto t_full = [&](int b) { return bar0 + 8u * (21 + b); };
  auto t_empty = [&](int b) { return bar0 + 8u * (25 + b); };
  auto s_full = [&](int b) { return bar0 + 8u * (29 + b); };
  auto p_full = [&](int b) { return bar0 + 8u * (32 + b); };
  auto buf_free = [&](int b) { return bar0 + 8u * (35 + b); };

  const int half = a.pool >> 1;
  const bool quarter = a.tiles_per_cta <= kQuarterTiles;
  const uint32_t hist_bytes = (uint32_t)(n_clu * kThr * 512);
  int ld_s = 0, ld_n = 0, ld_k = 0;   // producer: ring position, loads issued, K tiles of phase C among them
  uint32_t ld_ph = 1;
  // load n of the CTA: the tiles of phase S upwards, of phase V downwards (the last ones are the recent ones), then K
  // and V of phase C, K three tiles ahead: its S has a buffer by then, and a V slot is held until its P.V is done (in turn,
  // K(t+3) waited behind V(t+2) for P.V(t))
  const int n_loads = nS + nV + 2 * nC;
  auto load_next = [&]() -> bool {
    int tile = tile0 + ld_n;
    const CUtensorMap* map = &k_map;
    uint32_t bar = full_k(ld_s);
    if (ld_n >= nS + nV) {
      if (ld_k < min(nC, ld_n - nS - nV - ld_k + kCalBufs)) {
        tile = tile0 + ld_k++;
      } else {
        tile = tile0 + ld_n - nS - nV - ld_k;
        map = &v_map;
        bar = full_v(ld_s);
      }
    } else if (ld_n >= nS) {
      tile = tile0 + nV - 1 - (ld_n - nS);
    }
    if (!mbar_wait_far(&ctl, empty(ld_s), ld_ph, 61u)) return false;
    mbar_arrive_expect_tx(bar, kTileBytes);
#pragma unroll 1
    for (int h = 0; h < 2; ++h)
      tma_load_3d(ring + ld_s * kTileBytes + h * (kTileBytes / 2), map, bar, h * kHalfCols, tile * kTileKeys, unit);
    ++ld_n;
    if (++ld_s == a.stages) { ld_s = 0; ld_ph ^= 1u; }
    return true;
  };
  if (warp == kProducerWarp) {
    // barriers and the first loads, while the other warps set themselves up
    if (lane == 0) {
      ctl.abort = 0;
      ctl.status = a.status;
      next_row = 0;
    }
    // arrivals that complete a phase: one per CTA, one per consumer warp, or one
    for (int i = lane; i < kBars; i += 32) {
      const uint32_t bar = bar0 + 8u * i;
      const bool per_cta = bar == x_kept || bar == x_o;
      const bool per_warp = (bar >= t_empty(0) && bar <= t_empty(kAccBufs - 1)) || (bar >= p_full(0) && bar <= p_full(kCalBufs - 1));
      mbar_init(bar, per_cta ? n_clu : per_warp ? 16 : 1);
    }
    fence_mbar_init();
    __syncwarp();
    if (lane == 0) {
      // what the peers will push: armed before any of them can run past the cluster barrier below
      mbar_arrive_expect_tx(x_lse, (uint32_t)(n_clu * a.GW * 8));
      mbar_arrive_expect_tx(x_halo, (uint32_t)(n_clu * 4 + ((rank > 0) + (rank < n_clu - 1)) * half * 4));
      mbar_arrive_expect_tx(x_hist(0), hist_bytes);
      mbar_arrive_expect_tx(x_hist(1), hist_bytes);
      tma_prefetch_desc(&q_map);
      tma_prefetch_desc(&k_map);
    }
    __syncwarp();
    asm volatile("barrier.cta.arrive 2, %0;" ::"n"(kThreads) : "memory");   // the others need not wait for the loads
    pdl_wait();   // everything above ran beside the previous kernel's end; global memory from here on
    if (lane == 0) {
      if (nS + nV > 0) {
        // the window rows, as often as they fit on the lanes (rows beyond G * W arrive as zeros)
        mbar_arrive_expect_tx(q_full, kTileBytes);
#pragma unroll 1
        for (int c = 0; c < 1 << a.lg_rep; ++c)
#pragma unroll 1
          for (int h = 0; h < 2; ++h)
            tma_load_3d(q_base + h * (kTileBytes / 2) + c * ((kTileBytes / 2) >> a.lg_rep), &q_map, q_full, h * kHalfCols, 0,
                        unit);
      }
#pragma unroll 1
      while (ld_n < min(nS + nV, a.stages) && load_next()) {}
      if (rank == 0 && unit == 0) *a.status = 0u;
    }
    __syncwarp();
  }
  uint32_t tmem_base = 0u;
  if (warp != kProducerWarp) {
    if (warp == kMmaWarp) {
      tmem_alloc(smem_u32(&tmem_slot), 512);
      tmem_relinquish();
    }
    tc_fence_before_sync();
    asm volatile("barrier.cta.sync 2, %0;" ::"n"(kThreads) : "memory");
    tc_fence_after_sync();
    tmem_base = tmem_slot;
  }
  __syncwarp();
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");   // (fence_mbar_init releases the barriers)
  pdl_wait();

  // This CTA's share of the kept list is handed out to the warps that have time, eight rows at once, half a warp to a row:
  // to one warp from the selection on, to the consumers when they are done.  (By the one warp alone, 512 rows a CTA
  // took 8 us longer than everything else.)
  auto compact_rows = [&]() {
    const int per = (a.n_copy + n_clu - 1) / n_clu, i0 = min(a.n_copy, rank * per), i1 = min(a.n_copy, i0 + per);
    const int32_t* list = a.kept_idx + (size_t)unit * a.n_kept;
    constexpr int kRows = 4;
    const int sub = lane >> 4, chunk = lane & 15;
#pragma unroll 1
    while (true) {
      int at = 0;
      if (lane == 0) at = atomicAdd(&next_row, 2 * kRows);
      const int i = i0 + __shfl_sync(0xffffffffu, at, 0) + sub;
      if (i - sub >= i1) break;
      int t[kRows];
      uint4 k[kRows], v[kRows];
#pragma unroll
      for (int j = 0; j < kRows; ++j) {
        t[j] = i + 2 * j < i1 ? __ldcg(list + i + 2 * j) : -1;
        if (t[j] >= a.L) t[j] = -1;
      }
#pragma unroll
      for (int j = 0; j < kRows; ++j)
        if (t[j] >= 0) {
          const size_t src = ((size_t)unit * a.L + t[j]) * 16 + chunk;
          k[j] = __ldg(a.gather.K + src);
          v[j] = __ldg(a.gather.V + src);
        }
#pragma unroll
      for (int j = 0; j < kRows; ++j)
        if (t[j] >= 0) {
          const size_t dst = ((size_t)unit * a.gather.out_rows + i + 2 * j) * 16 + chunk;
          a.gather.K_out[dst] = k[j];
          a.gather.V_out[dst] = v[j];
        }
    }
  };
  if (warp == kProducerWarp) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      tma_prefetch_desc(&v_map);
      tma_prefetch_desc(&qc_map);
      bool ok = true;
#pragma unroll 1
      while (ok && ld_n < nS + nV) ok = load_next();
      if (nC > 0 && ok) {
        // the calibration rows replace the window rows once the last S^T is done
        ok = nS + nV == 0 || mbar_wait_far(&ctl, q_empty, 0, 62u);
        if (ok) {
          mbar_arrive_expect_tx(q_full, ((uint32_t)(2 * a.cal_rows) << a.lg_rep_c) * kLineBytes);
#pragma unroll 1
          for (int c = 0; c < 1 << a.lg_rep_c; ++c)
#pragma unroll 1
            for (int h = 0; h < 2; ++h)
              tma_load_4d(q_base + h * (kTileBytes / 2) + c * ((kTileBytes / 2) >> a.lg_rep_c), &qc_map, q_full,
                          h * kHalfCols, 0, 0, unit);
        }
#pragma unroll 1
        while (ok && ld_n < n_loads) ok = load_next();
      }
    }
    __syncwarp();
  } else if (__shfl_sync(0xffffffffu, warp, 0) == kMmaWarp) {
    // ------------------------------------------------------------ issuer of S and S^T (the warp as a whole, one lane issues)
    const uint32_t idesc = umma_idesc(128, 128, false, false), idesc_v = umma_idesc(128, a.n_pad, false, false);
    const uint64_t dq = smem_desc_sw128(q_base, 16u, 1024u), dk0 = smem_desc_sw128(ring, 16u, 1024u);
    const bool leader = elect_one();
    int s = 0, buf = 0;
    uint32_t k_ph = 0, t_ph = 1;   // k_ph: a phase bit per slot
    bool ok = nS + nV == 0 || __all_sync(0xffffffffu, mbar_wait_far(&ctl, q_full, 0, 63u));
#pragma unroll 1
    for (int j = 0; j < nS + nV && ok; ++j) {
      const bool votes = j >= nS;
      ok = mbar_wait_far(&ctl, full_k(s), (k_ph >> s) & 1u, 64u);
      ok = ok && mbar_wait_far(&ctl, t_empty(buf), t_ph, 65u);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after_sync();
      const uint32_t d = tmem_base + (uint32_t)(buf * 128);
      const uint64_t dk = desc_advance(dk0, (uint32_t)s * kTileBytes);
      const uint64_t da = votes ? dk : dq, db = votes ? dq : dk;
      const uint32_t id = votes ? idesc_v : idesc;
      if (leader) {
        umma_ss_imm<0>(d, da, db, id);
#pragma unroll
        for (int kk = 1; kk < kD / 16; ++kk)
          umma_ss_imm<1>(d, desc_advance(da, kmajor_step_bytes(kTileBytes / 2, kk)),
                         desc_advance(db, kmajor_step_bytes(kTileBytes / 2, kk)), id);
        umma_commit(t_full(buf));
        umma_commit(empty(s));
        if (j == nS + nV - 1) umma_commit(q_empty);
      }
      __syncwarp();
      k_ph ^= 1u << s;
      if (++s == a.stages) s = 0;
      if (++buf == kAccBufs) { buf = 0; t_ph ^= 1u; }
    }
    if (nC > 0 && ok) {
      ok = mbar_wait_far(&ctl, q_full, nS + nV > 0 ? 1u : 0u, 66u);
      // every accumulator of phase V has been read out: buf and t_ph are where the next job of that kind would go
#pragma unroll 1
      for (int b = 0; b < kAccBufs; ++b) {
        ok = ok && mbar_wait_far(&ctl, t_empty(buf), t_ph, 67u);
        if (++buf == kAccBufs) { buf = 0; t_ph ^= 1u; }
      }
      ok = __all_sync(0xffffffffu, ok);
      int b = 0;
      uint32_t b_ph = 1;
#pragma unroll 1
      for (int t = 0; t < nC && ok; ++t) {
        ok = mbar_wait_far(&ctl, full_k(s), (k_ph >> s) & 1u, 68u);
        ok = ok && mbar_wait_far(&ctl, buf_free(b), b_ph, 69u);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after_sync();
        const uint32_t d = tmem_base + (uint32_t)(b * 128);
        const uint64_t dk = desc_advance(dk0, (uint32_t)s * kTileBytes);
        if (leader) {
          umma_ss_imm<0>(d, dq, dk, idesc);
#pragma unroll
          for (int kk = 1; kk < kD / 16; ++kk)
            umma_ss_imm<1>(d, desc_advance(dq, kmajor_step_bytes(kTileBytes / 2, kk)),
                           desc_advance(dk, kmajor_step_bytes(kTileBytes / 2, kk)), idesc);
          umma_commit(s_full(b));
          umma_commit(empty(s));
        }
        __syncwarp();
        k_ph ^= 1u << s;
        s = (s + (t < kCalBufs - 1 ? 1 : 2)) % a.stages;   // (the V tiles between are the other issuer's)
        if (++b == kCalBufs) { b = 0; b_ph ^= 1u; }
      }
    }
  } else if (__shfl_sync(0xffffffffu, warp, 0) == kPvWarp) {
    // ------------------------------------------------------------ issuer of P.V
    const uint32_t idesc_o = umma_idesc(128, 128, false, true);
    const uint64_t dv0 = smem_desc_sw128(ring, kTileBytes / 2, 1024u);
    const bool leader = elect_one();
    const int n0 = nS + nV + min(nC, kCalBufs);   // the ring's position of the first V tile
    int s = n0 % a.stages, b = 0;
    uint32_t v_ph = 0, b_ph = 0;
    bool ok = true;
#pragma unroll 1
    for (int t = 0; t < nC && ok; ++t) {
      ok = mbar_wait_far(&ctl, full_v(s), (v_ph >> s) & 1u, 70u);
      ok = ok && mbar_wait_far(&ctl, p_full(b), b_ph, 71u);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after_sync();
      const uint64_t vd = desc_advance(dv0, (uint32_t)s * kTileBytes);
      const uint32_t pa = tmem_base + (uint32_t)(b * 128), od = tmem_base + kColO;
      if (leader) {
        // 16 keys = 8 columns of P per step; the P of a group's 32 keys lies at the first 16 of its 32 columns
        umma_ts(od, pa, vd, idesc_o, t > 0 ? 1u : 0u);
#pragma unroll
        for (int kk = 1; kk < kTileKeys / 16; ++kk)
          umma_ts_imm<1>(od, pa + (uint32_t)((kk >> 1) * 32 + (kk & 1) * 8),
                         desc_advance(vd, (uint32_t)kk * 16u * kLineBytes), idesc_o);
        umma_commit(buf_free(b));
        umma_commit(empty(s));
        if (t == nC - 1) umma_commit(o_full);
      }
      __syncwarp();
      v_ph ^= 1u << s;
      s = (s + (t + kCalBufs < nC ? 2 : 1)) % a.stages;
      if (++b == kCalBufs) { b = 0; b_ph ^= 1u; }
    }
  } else if (warp >= kGatherWarp) {
    // ------------------------------------------------------------ compaction of the retained rows: from the selection on
    if (!kGiven) {
      asm volatile("barrier.cta.sync 3, %0;" ::"n"(kConsumers + 32) : "memory");
      if (lane < n_clu) arrive_peer(peer_addr(x_kept, lane));
    }
    if (kGiven || mbar_wait_cluster(&ctl, x_kept, 0, 72u)) compact_rows();
    __syncwarp();
  } else {
    // ------------------------------------------------------------ consumers
    // (a wait that runs out raises the CTA's abort flag, all later waits return at once, and the warps walk on through
    // every block barrier: the results are not valid, but nothing hangs and nothing is written out of range)
    const int grp = warp >> 2, r128 = tid & 127, quad = warp & 3;
    const uint32_t lane_addr = tmem_base + ((uint32_t)(quad * 32) << 16);
    const f32x2 sc = pack2(a.scale2);
    const int hq0 = (unit / Hkv) * a.Hq + (unit % Hkv) * a.G;   // first query head of the unit
    auto block_sync = [&]() { asm volatile("barrier.cta.sync 1, %0;" ::"n"(kConsumers) : "memory"); };
    // the peers run: they may be pushed to
    auto peers_up = [&]() {
      __syncwarp();
      asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    };
    int buf = 0;
    uint32_t t_ph = 0;
    // n accumulators of phase S or V in turn, N columns of each.  (With the next one on its way to the registers while `fold`
    // works on the current one, in loops of two steps, the calls took longer: 8 units x 8192 keys 35.6 us instead of 33.5,
    // 8 x 2048 17.0 instead of 16.6.  Four warps a scheduler hide the wait, and the code is half as long.)
    auto drain = [&](auto n_tag, int n, uint32_t taddr, auto&& fold) __attribute__((always_inline)) {
      constexpr int N = decltype(n_tag)::value;
#pragma unroll 1
      for (int i = 0; i < n; ++i) {
        uint32_t r[N];
        mbar_wait_far(&ctl, t_full(buf), t_ph, 73u);
        __syncwarp();
        tc_fence_after_sync();
        tmem_issue(taddr + (uint32_t)(buf * 128), r);
        tmem_wait(r);
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(t_empty(buf));
        if (++buf == kAccBufs) { buf = 0; t_ph ^= 1u; }
        fold(r, i);
      }
    };

    // ---- S: statistics of the window rows.  With few rows there are copies of them on the lanes: a copy takes its own
    // part of the group's 32 columns, so that all four schedulers work (32 rows alone would sit on one of them).
    if (nS > 0) {
      const int rows = 128 >> a.lg_rep, row = r128 & (rows - 1), copy = r128 >> (7 - a.lg_rep);
      const int sub = 32 >> a.lg_rep, col0 = grp * 32 + copy * sub;
      const int lim = a.n_cand + row % a.W;                  // the last key the row may see (causal inside the window)
      const bool any = (quad * 32 & (rows - 1)) < a.GW;      // a warp without a row only hands the buffers on
      float2 ml = make_float2(-1e30f, 0.f);
      auto run = [&](auto n_tag) __attribute__((always_inline)) {
        constexpr int N = decltype(n_tag)::value;
        auto fold = [&](uint32_t (&r)[N], int i) __attribute__((always_inline)) {
          const int l0 = lim - ((tile0 + i) * kTileKeys + col0);
          if (!__all_sync(0xffffffffu, l0 >= N - 1)) {
#pragma unroll
            for (int e = 0; e < N; ++e)
              if (e > l0) r[e] = 0xff800000u;   // -inf
          }
          float m0 = -INFINITY, m1 = -INFINITY;
#pragma unroll
          for (int e = 0; e < N; e += 4) {
            m0 = fmaxf(m0, fmaxf(__uint_as_float(r[e]), __uint_as_float(r[e + 1])));
            m1 = fmaxf(m1, fmaxf(__uint_as_float(r[e + 2]), __uint_as_float(r[e + 3])));
          }
          const float m_new = fmaxf(ml.x, fmaxf(m0, m1) * a.scale2);
          const f32x2 nr = pack2(-m_new);
          f32x2 s0 = 0ull, s1 = 0ull;
#pragma unroll
          for (int e = 0; e < N; e += 4) {
            const f32x2 x0 = fma2(pack2(r[e], r[e + 1]), sc, nr), x1 = fma2(pack2(r[e + 2], r[e + 3]), sc, nr);
            s0 = add_exp2_pair<false>(s0, x0, e / 2);
            s1 = add_exp2_pair<false>(s1, x1, e / 2 + 1);
          }
          const float2 v = unpack2(add2(s0, s1));
          ml.y = fmaf(ml.y, ex2_approx(ml.x - m_new), v.x + v.y);
          ml.x = m_new;
        };
        drain(n_tag, nS, lane_addr + (uint32_t)col0, fold);
      };
      if (!any) {
#pragma unroll 1
        for (int i = 0; i < nS; ++i) {
          mbar_wait_far(&ctl, t_full(buf), t_ph, 73u);
          __syncwarp();
          if (lane == 0) mbar_arrive(t_empty(buf));
          if (++buf == kAccBufs) { buf = 0; t_ph ^= 1u; }
        }
      } else if (a.lg_rep == 0) run(std::integral_constant<int, 32>{});
      else if (a.lg_rep == 1) run(std::integral_constant<int, 16>{});
      else run(std::integral_constant<int, 8>{});
      xs[grp * 128 + r128] = ml;
      block_sync();
      peers_up();
      // The CTA's (max, sum) of a row, from the groups and copies, to every CTA of the cluster: a part per thread, the
      // parts of a row on neighbouring lanes.  (The maximum first, then one factor per part: factors on every level
      // would add up their errors.)
      {
        const int lg_parts = 2 + a.lg_rep, parts = 1 << lg_parts, r = tid >> lg_parts, part = lane & (parts - 1);
        const float2 v = xs[(part & 3) * 128 + (part >> 2) * rows + r];
        float M = v.x;
        for (int o = 1; o < parts; o <<= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
        float l = v.y * exp2_unbiased(v.x - M);
        for (int o = 1; o < parts; o <<= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (r < a.GW) {
          const uint32_t dst = smem_u32(lse_in + rank * 128 + r);
          for (int p = part; p < n_clu; p += parts) push_f32x2(peer_addr(dst, p), M, l, peer_addr(x_lse, p));
        }
      }
      mbar_wait_far(&ctl, x_lse, 0, 74u);
      __syncwarp();
      {
        // the cluster's row LSE, four threads to a row
        const int r = tid >> 2, sub = tid & 3;
        float2 v[kMaxClu / 4];
        float M = -1e30f;
#pragma unroll
        for (int q = 0; q < kMaxClu / 4; ++q) {
          v[q] = r < a.GW && q * 4 + sub < n_clu ? lse_in[(q * 4 + sub) * 128 + r] : make_float2(-1e30f, 0.f);
          M = fmaxf(M, v[q].x);
        }
        M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, 1));
        M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, 2));
        float l = 0.f;
#pragma unroll
        for (int q = 0; q < kMaxClu / 4; ++q) l += v[q].y * exp2_unbiased(v[q].x - M);
        l += __shfl_xor_sync(0xffffffffu, l, 1);
        l += __shfl_xor_sync(0xffffffffu, l, 2);
        if (sub == 0) {
          const float lse = r < a.GW ? (M + log2f(l)) * kLn2 : INFINITY;
          if (rank == 0 && r < a.GW) a.row_lse_out[(size_t)hq0 * a.W + r] = lse;
          lse_s[r] = lse;
          nlse2_s[r] = -lse * kLog2e;
        }
      }
    } else if (tid < kMaxRows) {
      const float lse = tid < a.GW ? a.row_lse[(size_t)hq0 * a.W + tid] : INFINITY;
      lse_s[tid] = lse;
      nlse2_s[tid] = -lse * kLog2e;
    }
    block_sync();

    if constexpr (kGiven) {
      // the listed rows of this CTA, and those that are no candidates, are not calibrated
      if (nS == 0) peers_up();
      for (int i = tid; i < nt * 4; i += kConsumers) {
        const int rest = n_own - i * 32;
        mask_s[i] = rest >= 32 ? 0u : rest <= 0 ? 0xffffffffu : 0xffffffffu << rest;
      }
      block_sync();
      const int32_t* const list = a.kept_idx + (size_t)unit * a.n_kept;
      for (int i = tid; i < a.n_kept; i += kConsumers) {
        const int at = list[i] - c0;   // (a caller's list may hold anything)
        if (at >= 0 && at < nt * kTileKeys) atomicOr(mask_s + (at >> 5), 1u << (at & 31));
      }
      block_sync();
    } else {
    // ---- V: votes of this CTA's keys.  Up to kQuarterTiles tiles the four groups share a tile, a quarter of the rows
    // each, and the parts meet in shared memory; beyond, a group takes every fourth tile alone.
#pragma unroll 1
    for (int i = tid; i < half; i += kConsumers) {   // the prompt's ends are padded with zeros
      if (rank == 0) stage[i] = 0.f;
      if (rank == n_clu - 1) stage[half + nt * kTileKeys + i] = 0.f;
    }
    float* const vote_g = a.vote + (size_t)unit * a.n_cand + c0;
    // sums of exp2 over N columns from column c on, against -lse2 of those rows
    auto sum_cols = [&](auto& r, int c, f32x2& acc0, f32x2& acc1) __attribute__((always_inline)) {
#pragma unroll
      for (int e = 0; e < (int)(sizeof(r) / 4); e += 4) {
        const ulonglong2 n4 = *reinterpret_cast<const ulonglong2*>(nlse2_s + c + e);
        const f32x2 x0 = fma2(pack2(r[e], r[e + 1]), sc, n4.x), x1 = fma2(pack2(r[e + 2], r[e + 3]), sc, n4.y);
        acc0 = add_exp2_pair<true>(acc0, x0, e / 2);
        acc1 = add_exp2_pair<true>(acc1, x1, e / 2 + 1);
      }
    };
    if (quarter) {
      auto run = [&](auto n_tag) __attribute__((always_inline)) {
        constexpr int N = decltype(n_tag)::value;
        float* const part = vparts + grp * (nt * kTileKeys) + r128;
        drain(n_tag, nV, lane_addr + (uint32_t)(grp * N), [&](uint32_t (&r)[N], int j) __attribute__((always_inline)) {
          f32x2 acc0 = 0ull, acc1 = 0ull;
          sum_cols(r, grp * N, acc0, acc1);
          const float2 acc = unpack2(add2(acc0, acc1));
          part[(nV - 1 - j) * kTileKeys] = acc.x + acc.y;
        });
      };
      if (a.n_pad == 128) run(std::integral_constant<int, 32>{});
      else if (a.n_pad == 64) run(std::integral_constant<int, 16>{});
      else run(std::integral_constant<int, 8>{});
    } else {
      // job nS + j of the CTA has accumulator (nS + j) % 4, so a group always meets the same one
#pragma unroll 1
      for (int j = 0; j < nV; ++j) {
        if ((j & 3) == grp) {
          mbar_wait_far(&ctl, t_full(buf), t_ph, 75u);
          __syncwarp();
          tc_fence_after_sync();
          f32x2 acc0 = 0ull, acc1 = 0ull;
          const uint32_t taddr = lane_addr + (uint32_t)(buf * 128);
          uint32_t ra[32], rb[32];
          tmem_ld32_issue(taddr, ra);
#pragma unroll 1
          for (int c = 0; c < a.n_pad; c += 64) {
            tmem_ld_wait(ra);
            if (c + 32 < a.n_pad) tmem_ld32_issue(taddr + c + 32, rb);
            sum_cols(ra, c, acc0, acc1);
            if (c + 32 < a.n_pad) {
              tmem_ld_wait(rb);
              if (c + 64 < a.n_pad) tmem_ld32_issue(taddr + c + 64, ra);
              sum_cols(rb, c + 32, acc0, acc1);
            }
          }
          tc_fence_before_sync();
          __syncwarp();
          if (lane < 4) mbar_arrive(t_empty(buf));   // (the barrier counts sixteen warps, four are at work)
          const float2 acc = unpack2(add2(acc0, acc1));
          const int idx = (nV - 1 - j) * kTileKeys + r128;
          const float v = idx < n_own ? acc.x + acc.y : 0.f;
          stage[half + idx] = v;
          if (idx < n_own) vote_g[idx] = v;
        }
        if (++buf == kAccBufs) { buf = 0; t_ph ^= 1u; }
      }
    }
    block_sync();
    if (nS == 0) peers_up();
    // the votes into the staging area, their ends to the neighbours
    const int n_stage = nt * kTileKeys;
#pragma unroll 1
    for (int i = tid; i < n_stage; i += kConsumers) {
      float v;
      if (quarter) {
        const float* p = vparts + i;
        v = i < n_own ? (p[0] + p[n_stage]) + (p[2 * n_stage] + p[3 * n_stage]) : 0.f;
        stage[half + i] = v;
        if (i < n_own) vote_g[i] = v;
      } else {
        v = i < n_own ? stage[half + i] : 0.f;
        if (i >= n_own) stage[half + i] = 0.f;
      }
      if (i < half && rank > 0)   // (every CTA but the last has tiles_per_cta tiles)
        push_u32(peer_addr(smem_u32(stage + half + a.tiles_per_cta * kTileKeys + i), rank - 1), __float_as_uint(v),
                 peer_addr(x_halo, rank - 1));
      if (i >= n_stage - half && rank < n_clu - 1)
        push_u32(peer_addr(smem_u32(stage + i - (n_stage - half)), rank + 1), __float_as_uint(v), peer_addr(x_halo, rank + 1));
    }
    block_sync();                       // the partial votes are read: the histograms may take their place
#pragma unroll 1
    for (int i = tid; i < kThr * 256 * kHistCopies / 4; i += kConsumers) reinterpret_cast<uint4*>(hist)[i] = make_uint4(0u, 0u, 0u, 0u);
    // a word to every CTA: its peer's histograms may come
    if (tid < n_clu) push_u32(peer_addr(smem_u32(&ccnt[0][rank][0]), tid), 0u, peer_addr(x_halo, tid));
    mbar_wait_far(&ctl, x_halo, 0, 76u);
    __syncwarp();

    // ---- select.  Key (warp w, row i, lane l) is number (w * rows + i) * 32 + l of this CTA: a warp owns a contiguous run.
    const int rows = (n_stage + kConsumers - 1) / kConsumers, key0 = warp * rows * 32 + lane;
    {
      const float fpool = (float)a.pool;
      float* const pl = a.pooled + (size_t)unit * a.n_cand + c0;
      auto pool_rows = [&](auto taps_tag) __attribute__((always_inline)) {
        constexpr int kTaps = decltype(taps_tag)::value;
#pragma unroll 1
        for (int idx = key0; idx < min(n_own, key0 + rows * 32); idx += 32) {
          float acc = 0.f;
          if constexpr (kTaps > 0) {
#pragma unroll
            for (int d = 0; d < kTaps; ++d) acc += stage[idx + d];
          } else {
#pragma unroll 1
            for (int d = 0; d < a.pool; ++d) acc += stage[idx + d];
          }
          const float p = acc / fpool;
          pl[idx] = p;
          keys[idx] = (unsigned)max(__float_as_int(p), 0);   // (a negative NaN ranks as zero)
        }
      };
      if (a.pool == 7) pool_rows(std::integral_constant<int, 7>{});
      else if (a.pool == 5) pool_rows(std::integral_constant<int, 5>{});
      else pool_rows(std::integral_constant<int, 0>{});
      __syncwarp();
    }
    block_sync();   // the histograms are clear
    unsigned prefix[kThr], k[kThr], thr[kThr], above[kThr], equal[kThr];
    unsigned last_bin[kThr];     // the bin that the last pass of a threshold chose, all of its keys taken or not
    bool open[kThr], last_all[kThr], last[kThr];
    // The first pass takes sixteen octaves below the highest value that the threshold can have, sixteen bins to each: the
    // pooled votes add up to the number of rows at most, so the k-th of them is G * W / k at most.  The bins at the ends hold
    // what lies beyond; a threshold there (a caller's row LSE may be anything) is searched from the top bit on.  Then
    // eight bits a pass: two passes are nearly always enough, where eight plain bits of exponent first took three.
    int base[kThr], rem[kThr];   // first bin of the first pass; bits not yet resolved
#pragma unroll
    for (int x = 0; x < kThr; ++x) {
      prefix[x] = 0u; thr[x] = 0u; above[x] = 0u; equal[x] = 0u; open[x] = true;
      last_bin[x] = 0u; last_all[x] = last[x] = false;
      k[x] = (unsigned)(a.k_sel + (x ? a.n_calib : 0));
      base[x] = (int)(__float_as_uint((float)a.GW / (float)k[x]) >> 19) - 254;
      rem[x] = 31;
    }
    // warp r: how many keys of CTA r lie above the bin that pass `pass` chose, and in it
    auto tally = [&](int pass) __attribute__((always_inline)) {
#pragma unroll
      for (int x = 0; x < kThr; ++x)
        if (last[x] && warp < n_clu) {
          const uint4 h = reinterpret_cast<const uint4*>(counts_of(pass & 1, x, warp))[lane];
          const unsigned w[4] = {h.x, h.y, h.z, h.w};
          unsigned g = 0u, e = 0u;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const unsigned n = j & 1 ? w[j >> 1] >> 16 : w[j >> 1] & 0xffffu, bj = 8u * lane + j;
            if (bj > last_bin[x]) g += n;
            if (bj == last_bin[x]) e += n;
          }
          g = __reduce_add_sync(0xffffffffu, g);
          e = __reduce_add_sync(0xffffffffu, e);
          above[x] += g + (last_all[x] ? e : 0u);
          equal[x] = last_all[x] ? 0u : e;
        }
    };
    int pass = 0;
#pragma unroll 1
    for (; pass < 5; ++pass) {
      const int b = pass & 1;
#pragma unroll 1
      for (int i = 0; i < rows; ++i) {
        const int idx = key0 + i * 32;
        const bool valid = idx < n_own;
        const unsigned key = valid ? keys[idx] : 0u;
#pragma unroll
        for (int x = 0; x < kThr; ++x)
          if (valid && open[x] && (key >> rem[x]) == prefix[x]) {   // (31: the sign bit, zero)
            const int bits = min(8, rem[x]);
            const unsigned bin = pass == 0 ? (unsigned)min(max((int)(key >> 19) - base[x], 0), 255)
                                           : (key >> (rem[x] - bits)) & ((1u << bits) - 1u);
            atomicAdd(hist + (x * 256 + bin) * kHistCopies + (lane & (kHistCopies - 1)), 1u);
          }
      }
      // (ahead of this CTA's push of the pass, without which no peer reaches the one that reuses the buffer)
      if (pass > 0) tally(pass - 1);
      block_sync();
      if (tid < kThr * 256) {
        // a bin per thread; eight lanes put their bins together and share out the cluster's CTAs
        uint4* h = reinterpret_cast<uint4*>(hist + tid * kHistCopies);
        const uint4 u = h[0], v = h[1];
        const unsigned n = (u.x + u.y + u.z + u.w) + (v.x + v.y + v.z + v.w);
        const unsigned two = n | (__shfl_down_sync(0xffffffffu, n, 1) << 16);
        uint4 eight;
        eight.x = __shfl_sync(0xffffffffu, two, lane & 24);
        eight.y = __shfl_sync(0xffffffffu, two, (lane & 24) + 2);
        eight.z = __shfl_sync(0xffffffffu, two, (lane & 24) + 4);
        eight.w = __shfl_sync(0xffffffffu, two, (lane & 24) + 6);
        const uint32_t dst = smem_u32(counts_of(b, tid >> 8, rank) + (tid & 248));
#pragma unroll 1
        for (int p = lane & 7; p < n_clu; p += 8) push_u32x4(peer_addr(dst, p), eight, peer_addr(x_hist(b), p));
        h[0] = h[1] = make_uint4(0u, 0u, 0u, 0u);
      }
      mbar_wait_far(&ctl, x_hist(b), (pass >> 1) & 1, 77u);
      __syncwarp();
      if (tid == 0 && pass < 3) mbar_arrive_expect_tx(x_hist(b), hist_bytes);   // for pass + 2
      // one warp per threshold: lane 0 owns the 8 highest bins; walk downwards until k keys are covered
      if (warp < kThr) {
        const int x = warp;
        unsigned c[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
        // (seven CTAs at a time: sums of 16 bits in pairs do not overflow)
#pragma unroll 1
        for (int r0 = 0; r0 < n_clu; r0 += 7) {
          uint4 sum = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
          for (int r = 0; r < 7; ++r)
            if (r0 + r < n_clu) {
              const uint4 h = reinterpret_cast<const uint4*>(counts_of(b, x, r0 + r))[31 - lane];
              sum.x += h.x; sum.y += h.y; sum.z += h.z; sum.w += h.w;
            }
          c[7] += sum.x & 0xffffu; c[6] += sum.x >> 16; c[5] += sum.y & 0xffffu; c[4] += sum.y >> 16;
          c[3] += sum.z & 0xffffu; c[2] += sum.z >> 16; c[1] += sum.w & 0xffffu; c[0] += sum.w >> 16;
        }
        unsigned p[8];
        p[0] = c[0];
#pragma unroll
        for (int j = 1; j < 8; ++j) p[j] = p[j - 1] + c[j];
        unsigned incl = p[7];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned n = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += n;
        }
        const unsigned kk = kSized && x == 1 ? k[kThr - 1] : k[0], before = incl - p[7];
        if (before < kk && incl >= kk) {
          unsigned run = before, skip = 0u, in_bin = c[0];
#pragma unroll
          for (int j = 0; j < 7; ++j)
            if (before + p[j] < kk) { run = before + p[j]; skip = j + 1; in_bin = c[j + 1]; }
          sel_bin[x] = 255u - 8u * lane - skip;
          sel_k[x] = kk - run;
          sel_all[x] = in_bin == kk - run;
        }
      }
      block_sync();
      bool more = false;
#pragma unroll
      for (int x = 0; x < kThr; ++x) {
        last[x] = open[x];
        if (!open[x]) continue;
        last_bin[x] = sel_bin[x];
        if (pass == 0 && (last_bin[x] == 0u || last_bin[x] == 255u)) {
          last[x] = false;
          more = true;
          continue;
        }
        last_all[x] = sel_all[x] != 0u;
        if (pass == 0) {
          rem[x] = 19;
          prefix[x] = last_bin[x] + base[x];
        } else {
          const int bits = min(8, rem[x]);
          rem[x] -= bits;
          prefix[x] = (prefix[x] << bits) | last_bin[x];
        }
        thr[x] = prefix[x] << rem[x];
        k[x] = sel_k[x];
        // every key of the bin is taken: so is every key at or above the bin's lowest bit pattern
        if (last_all[x]) k[x] = 0xffffffffu;
        open[x] = !last_all[x] && rem[x] > 0;
        more |= open[x];
      }
      if (!more) break;
    }
    tally(min(pass, 4));

    // ---- ordered compaction (ties to the lowest index): what the warps and CTAs ahead of this warp take
    unsigned before_gt[kThr], before_eq[kThr];
#pragma unroll
    for (int x = 0; x < kThr; ++x) {
      unsigned g = 0u, e = 0u;
#pragma unroll 1
      for (int i = 0; i < rows; ++i) {
        const int idx = key0 + i * 32;
        const unsigned key = idx < n_own ? keys[idx] : 0u;
        g += __popc(__ballot_sync(0xffffffffu, idx < n_own && key > thr[x]));
        e += __popc(__ballot_sync(0xffffffffu, idx < n_own && key == thr[x]));
      }
      if (lane == 0) {
        wcnt[x][warp][0] = g; wcnt[x][warp][1] = e;
        if (warp < n_clu) { ccnt[x][warp][0] = above[x]; ccnt[x][warp][1] = equal[x]; }
      }
    }
    block_sync();
#pragma unroll
    for (int x = 0; x < kThr; ++x) {
      unsigned g = lane < warp ? wcnt[x][lane & 15][0] : 0u, e = lane < warp ? wcnt[x][lane & 15][1] : 0u;
      if (lane < rank) { g += ccnt[x][lane & 15][0]; e += ccnt[x][lane & 15][1]; }
      before_gt[x] = __reduce_add_sync(0xffffffffu, g);
      before_eq[x] = __reduce_add_sync(0xffffffffu, e);
    }
    int32_t* const kept = a.kept_idx + (size_t)unit * a.n_kept;
    const unsigned lt = (1u << lane) - 1u;
#pragma unroll 1
    for (int i = 0; i < rows; ++i) {
      const int idx = key0 + i * 32, word = warp * rows + i;
      const bool valid = idx < n_own;
      const unsigned key = valid ? keys[idx] : 0u;
      const unsigned gm = __ballot_sync(0xffffffffu, valid && key > thr[0]);
      const unsigned em = __ballot_sync(0xffffffffu, valid && key == thr[0]);
      const unsigned gt_before = before_gt[0] + __popc(gm & lt), eq_before = before_eq[0] + __popc(em & lt);
      before_gt[0] += __popc(gm);
      before_eq[0] += __popc(em);
      const bool sel = valid && (key > thr[0] || (key == thr[0] && eq_before < k[0]));
      const unsigned pos = gt_before + min(eq_before, k[0]);
      if (sel && pos < (unsigned)a.k_sel) kept[pos] = c0 + idx;
      if (kSized) {
        // calibration size: the candidates among the first k_sel + n_calib that were not selected
        constexpr int y = kThr - 1;
        const unsigned em2 = __ballot_sync(0xffffffffu, valid && key == thr[y]);
        const bool in2 = valid && (key > thr[y] || (key == thr[y] && before_eq[y] + __popc(em2 & lt) < k[y]));
        before_eq[y] += __popc(em2);
        const unsigned w2 = ~__ballot_sync(0xffffffffu, in2 && !sel);
        if (lane == 0 && word < nt * 4) {
          mask_s[word] = w2;
          if (c0 + word * 32 < a.L) a.mask2[(size_t)unit * a.bitmap_words + (c0 >> 5) + word] = w2;
        }
      } else {
        const unsigned w1 = __ballot_sync(0xffffffffu, sel || !valid);
        if (lane == 0 && word < nt * 4) mask_s[word] = w1;
      }
    }
    // the window rows close the kept list
    if (rank == 0)
#pragma unroll 1
      for (int j = tid; j < a.L - a.n_cand; j += kConsumers) kept[a.k_sel + j] = a.n_cand + j;
    // the compacting warp tells the cluster: its release waits until the list has reached the L2, a thousand cycles
    asm volatile("barrier.cta.arrive 3, %0;" ::"n"(kConsumers + 32) : "memory");
    block_sync();
    }

    // ---- C: probabilities of the evicted keys (see calib_tc.cu); copies of the rows as in S
    const int rows_c = 128 >> a.lg_rep_c, row_c = r128 & (rows_c - 1), copy_c = r128 >> (7 - a.lg_rep_c);
    const bool valid_c = row_c < a.cal_rows, any_c = (quad * 32 & (rows_c - 1)) < a.cal_rows;
    f32x2 lsum = 0ull;
    {
      const int g = row_c / a.n_cal, cc = row_c - g * a.n_cal;
      const f32x2 nl2 = pack2(valid_c ? nlse2_s[g * a.W + a.W - a.n_cal + cc] : -INFINITY);
      // probabilities of this copy's N of the group's 32 keys -> bf16 pairs, the other copies' keys zero in this one
      auto run = [&](auto n_tag) __attribute__((always_inline)) {
        constexpr int N = decltype(n_tag)::value;
        const int first = copy_c * N;
        const uint32_t taddr = lane_addr + (uint32_t)(grp * 32);
        int b = 0;
        uint32_t b_ph = 0;
#pragma unroll 1
        for (int t = 0; t < nC; ++t) {
          uint32_t sv[N];
          mbar_wait_far(&ctl, s_full(b), b_ph, 78u);
          __syncwarp();
          tc_fence_after_sync();
          tmem_issue(taddr + (uint32_t)(b * 128 + first), sv);
          tmem_wait(sv);
          const uint32_t dst = taddr + (uint32_t)(b * 128), bar_p = p_full(b);
          if (++b == kCalBufs) { b = 0; b_ph ^= 1u; }
          const uint32_t w = mask_s[t * 4 + grp] >> first;
#pragma unroll
          for (int e = 0; e < N; e += 2) {
            const float2 p = unpack2(exp2_pair<true>(fma2(pack2(sv[e], sv[e + 1]), sc, nl2), e / 2));
            sv[e] = __float_as_uint(p.x);
            sv[e + 1] = __float_as_uint(p.y);
          }
          if (w != 0u) {
#pragma unroll
            for (int e8 = 0; e8 < N; e8 += 8)
              if ((w >> e8) & 0xffu) {
#pragma unroll
                for (int e = e8; e < e8 + 8; ++e)
                  if ((w >> e) & 1u) sv[e] = 0u;
              }
          }
          uint32_t packed[N / 2], out[16];
#pragma unroll
          for (int e = 0; e < N; e += 2) {
            lsum = add2(lsum, pack2(sv[e], sv[e + 1]));
            packed[e >> 1] = pack_bf16(__uint_as_float(sv[e]), __uint_as_float(sv[e + 1]));
          }
#pragma unroll
          for (int q = 0; q < 16; ++q) out[q] = N == 32 || q / (N / 2) == copy_c ? packed[q % (N / 2)] : 0u;
          tmem_st16(dst, out);
          tmem_st_wait();
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_p);
        }
      };
      if (!any_c) {
        // (the other rows' lanes; a probability in a row that is not read does no harm)
#pragma unroll 1
        for (int t = 0, b = 0, ph = 0; t < nC; ++t) {
          mbar_wait_far(&ctl, s_full(b), ph, 78u);
          __syncwarp();
          if (lane == 0) mbar_arrive(p_full(b));
          if (++b == kCalBufs) { b = 0; ph ^= 1; }
        }
      } else if (a.lg_rep_c == 0) run(std::integral_constant<int, 32>{});
      else if (a.lg_rep_c == 1) run(std::integral_constant<int, 16>{});
      else run(std::integral_constant<int, 8>{});
    }
    // ---- this CTA's partial O and row sums into the workspace, the copies of a row added up.  (Read from the peers' shared
    // memory instead, 128 rows of ten CTAs took 24 thousand cycles, 2.8 bytes a cycle and SM.)
    if (nC > 0) mbar_wait_far(&ctl, o_full, 0, 79u);
    __syncwarp();
    tc_fence_after_sync();
    if (any_c) {
      uint32_t ov[32];
      if (nC > 0) {
        tmem_ld32(lane_addr + kColO + (uint32_t)(grp * 32), ov);
      } else {
#pragma unroll
        for (int e = 0; e < 32; ++e) ov[e] = 0u;
      }
      uint4* const orow = reinterpret_cast<uint4*>(obuf + r128 * kOStride + grp * 32);
#pragma unroll
      for (int e = 0; e < 8; ++e) orow[e] = make_uint4(ov[4 * e], ov[4 * e + 1], ov[4 * e + 2], ov[4 * e + 3]);
    }
    const float2 lv = unpack2(lsum);
    l_s[grp][r128] = lv.x + lv.y;
    block_sync();
    {
      const size_t slot = ((size_t)unit * n_clu + rank) * a.cal_rows;
#pragma unroll 1
      for (int i = tid; i < a.cal_rows * 32; i += kConsumers) {
        const int row = i >> 5;
        float4 v = *reinterpret_cast<const float4*>(obuf + row * kOStride + 4 * lane);
#pragma unroll 1
        for (int c = 1; c < 1 << a.lg_rep_c; ++c) {
          const float4 u = *reinterpret_cast<const float4*>(obuf + (c * rows_c + row) * kOStride + 4 * lane);
          v.x += u.x; v.y += u.y; v.z += u.z; v.w += u.w;
        }
        if (a.lg_rep_c > 0 && __any_sync(0xffffffffu, isnan(v.x) || isnan(v.y) || isnan(v.z) || isnan(v.w))) {   // (a warp to a row)
          const int wrow = row / a.n_cal * a.W + a.W - a.n_cal + row % a.n_cal;
          float l = 0.f;
          for (int c = 0; c < 1 << a.lg_rep_c; ++c)
            for (int q = 0; q < kGroups; ++q) l += l_s[q][c * rows_c + row];
          const size_t first = ((size_t)unit * a.L + c0) * kD;
          v = refold_nonfinite(v, a.Q_obs + ((size_t)hq0 * a.W + wrow) * kD,
                               reinterpret_cast<const __nv_bfloat16*>(a.gather.K) + first,
                               reinterpret_cast<const __nv_bfloat16*>(a.gather.V) + first, min(nC * kTileKeys, a.L - c0), mask_s,
                               a.scale2, nlse2_s[wrow], l, lane);
        }
        __stcg(reinterpret_cast<float4*>(a.o_part + slot * kD) + i, v);
      }
      if (tid < a.cal_rows) {
        float l = 0.f;
#pragma unroll 1
        for (int c = 0; c < 1 << a.lg_rep_c; ++c)
#pragma unroll
          for (int q = 0; q < kGroups; ++q) l += l_s[q][c * rows_c + tid];
        __stcg(a.l_part + slot + tid, l);
      }
    }
    block_sync();
    if (tid < n_clu) arrive_peer(peer_addr(x_o, tid));
    mbar_wait_cluster(&ctl, x_o, 0, 80u);
    __syncwarp();
    // ---- a warp per calibration row: O_c = O / l, LSE_c = lse + log l (zeros and -inf when nothing was evicted), C_q
#pragma unroll 1
    for (int row = rank + warp * n_clu; row < a.cal_rows; row += 16 * n_clu) {
      const int g = row / a.n_cal, cc = row - g * a.n_cal, wrow = g * a.W + a.W - a.n_cal + cc;
      const size_t slot0 = (size_t)unit * n_clu * a.cal_rows + row;
      const uint2 cq = reinterpret_cast<const uint2*>(a.Q_obs + ((size_t)hq0 * a.W + wrow) * kD)[lane];
      float l = lane < n_clu ? __ldcg(a.l_part + slot0 + (size_t)lane * a.cal_rows) : 0.f;
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
      float4 v[kMaxClu];
#pragma unroll
      for (int p = 0; p < kMaxClu; ++p)
        v[p] = p < n_clu ? __ldcg(reinterpret_cast<const float4*>(a.o_part + (slot0 + (size_t)p * a.cal_rows) * kD) + lane)
                         : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int p = 0; p < kMaxClu; ++p) { acc.x += v[p].x; acc.y += v[p].y; acc.z += v[p].z; acc.w += v[p].w; }
      l = warp_sum(l);
      float4 out = make_float4(0.f, 0.f, 0.f, 0.f);
      float lse = -INFINITY;
      if (l > 0.f) {
        const float inv = 1.f / l;
        out = make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
        lse = lse_s[wrow] + logf(l);
      }
      const size_t dst = (size_t)hq0 * a.n_cal + row;
      reinterpret_cast<float4*>(a.O_c + dst * kD)[lane] = out;
      if (lane == 0) a.LSE_c[dst] = lse;
      reinterpret_cast<uint2*>(a.C_q + dst * kD)[lane] = cq;
    }
    if (kGiven || mbar_wait_cluster(&ctl, x_kept, 0, 81u)) compact_rows();
  }

  // ---------------------------------------------------------------- teardown (every path)
  __syncwarp();
  if (warp >= kProducerWarp) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // (the first one)
  if (ctl.abort) {
#pragma unroll 1
    for (int i = 0; i < 50; ++i) __nanosleep(20000);  // let TMA copies still in flight land
  }
  tc_fence_before_sync();
  __syncthreads();
  pdl_trigger();
  if (warp == kMmaWarp) tmem_dealloc(tmem_base, 512);
  // a CTA leaves when nobody writes to its shared memory any more
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}


struct ClusterPlan {
  int tiles_per_cta, n_clu, stages, stage_off, keys_off, mask_off, smem;
  bool copy_behind;   // the retained rows are compacted by a kernel of their own
};

int round_up(int x, int to) { return (x + to - 1) / to * to; }

// Shared memory of a plan with the given tiles per CTA; false where the ring would be too short.
bool lay_out(const CompressGeom& g, bool stats, int tiles_per_cta, ClusterPlan* p) {
  const int thr = g.sized ? 2 : 1;
  p->tiles_per_cta = tiles_per_cta;
  const int n_tiles = (g.L + kTileKeys - 1) / kTileKeys;
  p->n_clu = (n_tiles + tiles_per_cta - 1) / tiles_per_cta;
  int area = thr * (256 * kHistCopies * 4 + 2 * p->n_clu * 512);
  if (stats) area = std::max(area, (kGroups + p->n_clu) * 1024);
  if (tiles_per_cta <= kQuarterTiles) area = std::max(area, kGroups * tiles_per_cta * kTileKeys * 4);
  p->stage_off = round_up(area, 16);
  p->keys_off = p->stage_off + round_up((tiles_per_cta * kTileKeys + 2 * (g.pool >> 1)) * 4, 16);
  p->mask_off = p->keys_off + tiles_per_cta * kTileKeys * 4;
  const int scratch = p->mask_off + tiles_per_cta * 16;
  p->stages = std::min((kSmemMax - 1024 - kTileBytes - scratch) / kTileBytes, kMaxStages);
  p->smem = 1024 + kTileBytes * (1 + p->stages) + scratch;
  return p->stages >= kMinStages;   // (the partial O takes the place of three tiles)
}

void launch_config(int n_clu, int units, int smem, cudaStream_t st, cudaLaunchConfig_t& cfg, cudaLaunchAttribute (&attr)[2]) {
  cfg = cudaLaunchConfig_t{};
  cfg.gridDim = dim3(n_clu, units);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = n_clu;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
}

template <bool kSized, bool kGiven>
cudaError_t setup() {
  static OncePerDevice granted, wide;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = grant_smem(compress_cluster_kernel<kSized, kGiven>, kSmemMax, granted);
  if (e != cudaSuccess) return e;
  const bool slot = dev >= 0 && dev < 64;
  if (slot && wide[dev].load(std::memory_order_acquire)) return cudaSuccess;
  e = cudaFuncSetAttribute(compress_cluster_kernel<kSized, kGiven>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess && slot) wide[dev].store(true, std::memory_order_release);
  return e;
}

// Clusters of n_clu CTAs that the current device runs at the same time (the shape of its processor clusters decides).
int resident_clusters(int n_clu) {
  static std::atomic<int> known[64][kMaxClu + 1];   // 0: not asked yet, else 1 + clusters
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  int n = known[dev][n_clu].load(std::memory_order_acquire);
  if (n == 0) {
    if (setup<false, false>() != cudaSuccess) return 0;
    int active = 0;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    launch_config(n_clu, 1, kSmemMax, nullptr, cfg, attr);
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&active, compress_cluster_kernel<false, false>, &cfg) != cudaSuccess) {
      cudaGetLastError();   // no such cluster on this device
      active = 0;
    }
    n = 1 + active;
    known[dev][n_clu].store(n, std::memory_order_release);
  }
  return n - 1;
}

template <bool kSized, bool kGiven>
cudaError_t launch_kernel(const ClusterArgs& a, const ClusterPlan& p, int units, const CUtensorMap& qm, const CUtensorMap& qcm,
                          const CUtensorMap& km, const CUtensorMap& vm, cudaStream_t st) {
  cudaError_t e = setup<kSized, kGiven>();
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  launch_config(p.n_clu, units, p.smem, st, cfg, attr);
  e = cudaLaunchKernelEx(&cfg, compress_cluster_kernel<kSized, kGiven>, qm, qcm, km, vm, a);
  if (e != cudaSuccess) return e;
  count_launch(1);
  return cudaGetLastError();
}

// The fewest tiles per CTA with which every unit has its cluster at once; false where the kernel does not cover the
// shape or the separate kernels are the faster way.  What a call costs, in microseconds: here a chain and each tile of a CTA, there
// a chain, each tile of an SM, where all SMs have a share (here those that no cluster fits on are idle), and the selection of a long
// unit; the compaction costs both alike, but for 3 where it is a kernel behind this one.  The constants for the separate kernels are
// those with which the fewest of 333 calls, drawn wide and timed both ways on inputs in L2 and not, took the slower way; the margin of
// 4 % is from 300 more, of which one is still slower here (80 units x 2745 keys 66.4 and 69.8; 66.8 and 67.4 from memory).  (Constants fitted
// to 30 shapes, without a margin, took 80 x 3109 x 128 rows with the caller's row LSE, 59 here and 54 there, and 4 x 56877 for a given list,
// 92 and 81.)  Measured, us, separate and here: 8 units x 1100 keys x 128 rows 32.0 and 18, x 8192 44 and 32, x 16384 62 and
// 47, x 32768 84 and 81; 2 units x 24000 56 and 43; 16 x 16384 81 and 73; 32 x 2048 46 and 26, x 20000 146 and 129; with the caller's
// row LSE 16 x 24576 80 and 76, 64 x 12288 135 and 122.  For a given kept list 8 x 1000 24 and 12, x 8192 31 and 21, x 45000 77 and
// 66, 2 x 24000 41 and 28, 64 x 8192 100 and 77; with the caller's row LSE 8 x 8192 22 and 14, 16 x 32768 65 and 54.
bool plan_cluster(const CompressGeom& g, bool stats, bool given, ClusterPlan* p) {
  if (g.keep_all || g.n_cand < 1 || g.G * g.W > kMaxRows || g.pool >> 1 > kHaloMax) return false;
  if (g.sized && g.n_calib == 0) return false;
  const int n_tiles = (g.L + kTileKeys - 1) / kTileKeys;
  // the CTAs' partial O lie where the separate calibration's would
  int gpb, n_cblocks, tpc, max_slots;
  size_t parts;
  calib_tc_plan(g, &gpb, &n_cblocks, &tpc, &max_slots, &parts);
  for (int t = (n_tiles + kMaxClu - 1) / kMaxClu; t <= kMaxTiles; ++t) {
    const int n_clu = (n_tiles + t - 1) / t;
    if (g.units > resident_clusters(n_clu) || (size_t)g.units * n_clu > parts) continue;
    const double tiles = (double)g.units * n_tiles / kSms;
    const double here = given ? (stats ? 10.5 + 1.55 * t : 8.7 + 0.95 * t) : 13.0 + (stats ? 2.58 : 1.9) * t;
    const double there = given ? 25.0 + (stats ? 2.72 : 1.2) * tiles : 35.0 + (stats ? 3.6 : 1.76) * tiles + g.L * 1.5e-4;
    p->copy_behind = g.n_kept > kCopyRows * n_clu;
    return 1.04 * (here + (p->copy_behind ? 3.0 : 0.0)) < there && lay_out(g, stats, t, p);
  }
  return false;
}

}  // namespace

// The whole step in one launch (two with many retained rows), or (`given`) the calibration and compaction for the kept list in
// kept_idx; *taken is false (and nothing launched) where the separate kernels are to be used.
cudaError_t launch_compress_cluster(const CompressGeom& g, const CompressWs& ws, const void* Q_obs, const void* K, const void* V,
                                    const float* row_lse, char* wsp, int32_t* kept_idx, float* O_c, float* LSE_c, void* C_q,
                                    const GatherArgs& gather, bool given, bool* taken, cudaStream_t st) {
  ClusterPlan p;
  *taken = plan_cluster(g, row_lse == nullptr, given, &p);
  if (!*taken) return cudaSuccess;
  ClusterArgs a{};
  a.Hq = g.Hq; a.G = g.G; a.W = g.W; a.L = g.L; a.n_cand = g.n_cand; a.n_cal = g.n_cal;
  a.GW = g.G * g.W; a.cal_rows = g.G * g.n_cal;
  a.n_tiles = (g.L + kTileKeys - 1) / kTileKeys;
  a.tiles_per_cta = p.tiles_per_cta; a.n_clu = p.n_clu; a.stages = p.stages;
  auto copies = [](int rows) { return rows <= 32 ? 2 : rows <= 64 ? 1 : 0; };
  a.lg_rep = copies(a.GW);
  a.lg_rep_c = copies(a.cal_rows);
  a.n_pad = 128 >> a.lg_rep;
  a.pool = g.pool; a.k_sel = g.k_sel; a.n_kept = g.n_kept; a.n_calib = g.n_calib; a.bitmap_words = g.bitmap_words;
  a.stage_off = p.stage_off; a.keys_off = p.keys_off; a.mask_off = p.mask_off;
  a.scale2 = g.scale2;
  a.row_lse = row_lse;
  a.row_lse_out = (float*)(wsp + ws.row_lse);
  a.vote = (float*)(wsp + ws.vote);
  a.pooled = (float*)(wsp + ws.pooled);
  a.mask2 = (uint32_t*)(wsp + ws.bitmap2);
  a.kept_idx = kept_idx;
  a.Q_obs = (const __nv_bfloat16*)Q_obs;
  a.O_c = O_c; a.LSE_c = LSE_c; a.C_q = (__nv_bfloat16*)C_q;
  a.o_part = (float*)(wsp + ws.calib_o);
  a.l_part = (float*)(wsp + ws.calib_l);
  a.gather = gather;
  a.status = (unsigned*)(wsp + ws.status);
  CUtensorMap qm, qcm, km, vm;
  const uint64_t qd[2] = {(uint64_t)a.GW, (uint64_t)g.units}, qs[2] = {256, (uint64_t)a.GW * 256};
  const uint32_t qb[2] = {128u >> a.lg_rep, 1};
  // calibration rows: [head dim][c < n_cal][g < G][unit], starting at observation row W - n_cal
  const uint64_t cd[3] = {(uint64_t)g.n_cal, (uint64_t)g.G, (uint64_t)g.units};
  const uint64_t cs[3] = {256, (uint64_t)g.W * 256, (uint64_t)g.G * g.W * 256};
  const uint32_t cb[3] = {(uint32_t)g.n_cal, (uint32_t)g.G, 1};
  const uint64_t kd[2] = {(uint64_t)g.L, (uint64_t)g.units}, ks[2] = {256, (uint64_t)g.L * 256};
  const uint32_t kb[2] = {(uint32_t)kTileKeys, 1};
  if (!make_tensor_map_bf16(&qm, Q_obs, 3, qd, qs, qb) ||
      !make_tensor_map_bf16(&qcm, (const char*)Q_obs + (size_t)(g.W - g.n_cal) * 256, 4, cd, cs, cb) ||
      !make_tensor_map_bf16(&km, K, 3, kd, ks, kb) || !make_tensor_map_bf16(&vm, V, 3, kd, ks, kb))
    return cudaErrorInvalidValue;
  a.n_copy = p.copy_behind ? 0 : g.n_kept;
  cudaError_t e = given     ? launch_kernel<false, true>(a, p, g.units, qm, qcm, km, vm, st)
                  : g.sized ? launch_kernel<true, false>(a, p, g.units, qm, qcm, km, vm, st)
                            : launch_kernel<false, false>(a, p, g.units, qm, qcm, km, vm, st);
  if (e == cudaSuccess && p.copy_behind) e = launch_gather(g, K, V, kept_idx, gather.K_out, gather.V_out, st);
  return e;
}

}  // namespace calidrop
