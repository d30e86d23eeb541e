// Decode-time attention over the compacted retained cache, merged with the calibration term.
//
// One launch covers: the append of the step's new K/V row, a split-K flash-decode over the
// retained rows with the G query heads of a kv group packed into one MMA tile (so every K/V
// byte is read once for all of them), the cosine similarity of the query with the stored
// calibration queries, the threshold gate, and the merge of Eq. 1-2.  The work is bound by
// HBM traffic (about 2G flop per byte), so the contraction uses the warp-level mma.sync path;
// what matters is how the bytes get to the SM and how short the chain after the last byte is.
//
// Grid: (split, batch*kv-head, layer); the splits of one (unit, layer) form thread-block
// clusters of 1, 2, 4, 8 or 16 CTAs.  A CTA has one producer warp and eight stream warps.  The
// producer moves the CTA's slice of K and V through a ring of six 64-row slots with TMA
// (128-byte swizzle, so ldmatrix is conflict-free and no load instruction per 16 bytes is
// spent on the stream); each slot is consumed by four stream warps, 16 rows each, with their
// own online softmax.  Launches of more (unit, layer) pairs than SMs take smaller CTAs, several to an
// SM, one per pair (ShapePair, ShapeNarrow).  The products are taken transposed, keys on the 16-row side of the MMA and
// the (at most eight) heads on its 8-column side, so that no half of a tile is padding:
//   S^T[16 keys x 8 heads]   = K_blk[16 x 128] . Q^T[128 x 8]          (8 MMAs)
//   O^T[128 dims x 8 heads] += V_blk^T[128 x 16 keys] . P^T[16 x 8]     (8 MMAs)
// The splits are combined inside the cluster through distributed shared memory: every CTA
// finishes a slice of the 128 output dimensions for all heads of the group, and each CTA pushes
// its partial of a slice into the shared memory of the slice's owner with asynchronous stores that
// report their bytes to an mbarrier there, so that every CTA waits for its own data only and then
// reduces local data.  Where few units share a very long cache (see
// plan_decode) a unit gets up to eight clusters;
// each writes its combined partial, its (max, sum) pair and its best similarity to the workspace, and
// the CTA that takes the last ticket of the unit's arrival counter merges them and resets the counter.
//
// A launch moves only tens of MB, so its latency chain matters as much as its bandwidth:
//   * the launch carries the programmatic-serialisation attribute and the kernel, first thing,
//     prefetches the head of its K/V slice into L2, ahead of the dependency wait;
//   * everything that does not need the predecessor's results (barrier setup, the address
//     arithmetic of all later loads) is done ahead of the wait as well;
//   * the similarity work (which needs only q and C_q) runs while the first slots are in flight,
//     and each CTA's best (similarity, row) pairs are pushed to the others early; the producer warp,
//     idle once the last slot is on its way, settles the calibration row meanwhile, and the chosen
//     O_c elements are fetched while the partial outputs are combined;
//   * the cache stream carries an evict-first L2 hint, the calibration state an evict-last hint.
#include <cooperative_groups.h>

#include <atomic>

#include "common.cuh"
#include "internal.h"
#include "tc_common.cuh"

namespace calidrop {

namespace {

namespace cg = cooperative_groups;

constexpr int kBlkRows = 16;                        // rows of one warp's MMA block
constexpr int kWideRows = 64;                       // rows of the boxes of whole slots in the wide shape
// The shape of a CTA: ring slots of kRows rows, each consumed by kRows / 16 warps, kWarps stream warps in two groups on
// alternate slots, kCtas CTAs per SM.
template <int kSlots_, int kRows_, int kCtas_, int kClu_, bool kHalf_ = false>
struct Shape {
  static constexpr int kSlots = kSlots_, kRows = kRows_, kCtas = kCtas_;
  static constexpr int kClu = kClu_;                // the most CTAs of a cluster
  static constexpr bool kHalf = kHalf_;             // whole slots by a copy per half of the columns (see DecodeCommon)
  static constexpr int kSubs = kRows / kBlkRows;    // warps per slot
  static constexpr int kStreamWarps = 2 * kSubs;
  static constexpr int kThreads = (kStreamWarps + 1) * 32;   // the last warp is the producer
  static constexpr int kPlaneBytes = kRows * 128;   // rows x 64 columns of bf16
  static constexpr int kSlotBytes = 4 * kPlaneBytes;         // K low / K high / V low / V high column halves
  static constexpr int kSmemBytes = kSlots * kSlotBytes + 1024;   // + slack for the 1024-byte alignment
};
template <bool kHalf>
using ShapeWide = Shape<6, kWideRows, 1, 8, kHalf>;     // a launch with one CTA per SM at most: 192 KB
template <bool kHalf>
using ShapeCluster16 = Shape<6, kWideRows, 1, 16, kHalf>;  // few units with a longer cache (see plan_decode)
template <bool kHalf>
using ShapePair = Shape<3, kWideRows, 2, 1, kHalf>;     // a launch with up to two CTAs per SM: 96 KB
using ShapeNarrow = Shape<3, 32, 4, 1>;                 // more than that: 48 KB, four CTAs per SM
constexpr int kWoStride = kD + 4;  // row stride of the per-warp partial outputs: heads land in distinct banks
constexpr long long kWaitLimitCycles = 2000000000ll;  // about a second: a wait this long has failed

// The K or the V part of a slot, as the copies leave it: the two halves of the columns as planes of 128-byte lines in the
// 128-byte swizzle, over the whole slot where one copy brings it (64 rows), else a pair of planes for every 16 rows.
struct Planes {
  uint32_t block, half;   // bytes from a 16-row block to the next, and from the first half of a block to its second
};
template <class S>
__device__ __forceinline__ Planes planes_of(bool whole) {
  return whole ? Planes{kBlkRows * 128, S::kPlaneBytes} : Planes{2 * kBlkRows * 128, kBlkRows * 128};
}
// Byte offset of 16-byte chunk `chunk` (0..15) of row `row` (0..15) of a block.
__device__ __forceinline__ uint32_t block_off(const Planes& p, int row, int chunk) {
  return (uint32_t)(chunk >> 3) * p.half + (uint32_t)(row * 128 + (((chunk & 7) ^ (row & 7)) << 4));
}

__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t x) {
  uint32_t y;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
  return y;
}

// ---- mbarrier / TMA helpers (every copy lands in the shared memory of the CTA that issued it)
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "selp.u32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait: when it runs out the CTA's abort flag is raised, the workspace's error word is
// set and every later wait of the CTA returns at once; the CTA still walks through all its
// barriers, so nothing hangs, but its output is not valid.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                          unsigned* status, unsigned code) {
  if (mbar_try_wait(bar, parity)) return true;
  long long t0 = 0;
  unsigned polls = 0;
  while (!mbar_try_wait(bar, parity)) {
    if ((++polls & 255u) == 0u) {
      if (*abort_flag) return false;
      const long long now = clock64();
      if (t0 == 0) t0 = now;
      if (now - t0 > kWaitLimitCycles) {
        *abort_flag = 1;
        atomicCAS(status, 0u, code);
        return false;
      }
    }
  }
  return true;
}
// The same wait without the shortcut on the CTA's abort flag: only its own time limit ends it early.
// For waits that must be sat out even in a CTA that is giving up, because other CTAs still write
// into (or read from) this CTA's shared memory until the awaited phase completes.
__device__ __forceinline__ bool mbar_wait_sit_out(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                                  unsigned* status, unsigned code) {
  long long t0 = 0;
  unsigned polls = 0;
  while (!mbar_try_wait(bar, parity)) {
    if ((++polls & 255u) == 0u) {
      const long long now = clock64();
      if (t0 == 0) t0 = now;
      if (now - t0 > kWaitLimitCycles) {
        *abort_flag = 1;
        atomicCAS(status, 0u, code);
        return false;
      }
    }
  }
  return true;
}
// Rows from row on of a unit: both halves of the head dimension, or half `h` alone where the map's box has one.
__device__ __forceinline__ void tma_load_rows(uint32_t dst, const CUtensorMap* map, uint32_t bar, int row, int unit,
                                              uint64_t pol, int h = 0) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint "
      "[%0], [%1, {%3, %4, %5, %7}], [%2], %6;"
      ::"r"(dst), "l"(map), "r"(bar), "r"(0), "r"(row), "r"(unit), "l"(pol), "r"(h)
      : "memory");
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, unsigned bytes, uint32_t bar, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(bar), "l"(pol)
      : "memory");
}

// L2 eviction policies.  The retained cache is read once per call and is far larger than what the
// next call on the same state finds in L2 again, so its lines are marked to go first; the
// calibration state (C_q, the chosen O_c rows, LSE_c) is small and read by every call, so its
// lines are marked to stay.  With that the similarity loads are L2 hits and do not queue behind
// the stream in the memory system.
__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint4 ldg_keep(const uint4* ptr, uint64_t pol) {
  uint4 v;
  asm volatile("ld.global.nc.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(ptr), "l"(pol));
  return v;
}
__device__ __forceinline__ float ldg_keep(const float* ptr, uint64_t pol) {
  float v;
  asm volatile("ld.global.nc.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(ptr), "l"(pol));
  return v;
}

// Shared-memory address of `local` in CTA `rank` of the cluster, and an 8-byte store to such an
// address that reports its bytes to an mbarrier of the same CTA when it lands.
__device__ __forceinline__ uint32_t cluster_addr(uint32_t local, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
  return r;
}
__device__ __forceinline__ void push_f32x2(uint32_t remote, float x, float y, uint32_t remote_bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(remote),
               "f"(x), "f"(y), "r"(remote_bar)
               : "memory");
}

__device__ __forceinline__ void push_f32x4(uint32_t remote, float4 v, uint32_t remote_bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(
                   remote),
               "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(remote_bar)
               : "memory");
}
__device__ __forceinline__ void push_u64(uint32_t remote, unsigned long long x, uint32_t remote_bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.u64 [%0], %1, [%2];" ::"r"(remote), "l"(x),
               "r"(remote_bar)
               : "memory");
}

struct RhoLoad {
  uint4 q0, q1, c0, c1;
};

__device__ __forceinline__ void rho_accumulate(const uint4& q, const uint4& c, float& dot, float& qq, float& cc) {
  const uint32_t qw[4] = {q.x, q.y, q.z, q.w}, cw[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float a0 = bf16_lo(qw[j]), a1 = bf16_hi(qw[j]);
    const float b0 = bf16_lo(cw[j]), b1 = bf16_hi(cw[j]);
    dot = fmaf(a0, b0, fmaf(a1, b1, dot));
    qq = fmaf(a0, a0, fmaf(a1, a1, qq));
    cc = fmaf(b0, b0, fmaf(b1, b1, cc));
  }
}
__device__ __forceinline__ void rho_accumulate(const RhoLoad& r, float& dot, float& qq, float& cc) {
  rho_accumulate(r.q0, r.c0, dot, qq, cc);
  rho_accumulate(r.q1, r.c1, dot, qq, cc);
}

// Order-preserving map of a float onto unsigned integers; with the row index in the low word,
// one 64-bit max picks the highest similarity and, among equals, the largest row index.
__device__ __forceinline__ unsigned long long rank_key(float rho, int c) {
  unsigned u = __float_as_uint(rho);
  u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
  return ((unsigned long long)u << 32) | (unsigned)c;
}
__device__ __forceinline__ float rank_key_value(unsigned long long k) {
  unsigned u = (unsigned)(k >> 32);
  u = (u & 0x80000000u) ? (u & 0x7fffffffu) : ~u;
  return __uint_as_float(u);
}

__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Gate and merge (Eq. 1-2) of `kN` neighbouring output elements of a head: (acc, M, Lsum) is the unnormalised partial of
// the retained cache in the log2 domain, best the chosen (similarity, calibration row) key.
template <int kN>
__device__ __forceinline__ void merge_store(const DecodeCommon& a, const DecodeLayerPtrs& P, int hq, int d,
                                            const float (&acc)[kN], float M, float Lsum, unsigned long long best,
                                            float lse_c, const float (&oc)[kN]) {
  const int cs = (int)(unsigned)(best & 0xffffffffull);
  const float rho = rank_key_value(best);
  float outv[kN];
#pragma unroll
  for (int e = 0; e < kN; ++e) outv[e] = __fdividef(acc[e], Lsum);  // O_a
  float lse2 = M + __log2f(Lsum);      // LSE_a (log2 domain)
  const bool apply = (a.always_apply || rho > a.theta2) && (lse_c > -INFINITY);
  if (apply) {
    // alpha_i = e^{LSE_a - LSE}, alpha_j = e^{LSE_c - LSE}; out = alpha_i O_a + alpha_j O_c
    const float lc2 = lse_c * kLog2e;
    const float mx = fmaxf(lse2, lc2);
    const float ea = ex2_approx(lse2 - mx), ec = ex2_approx(lc2 - mx);
    const float inv = __fdividef(1.f, ea + ec);  // the sum is in [1, 2]
#pragma unroll
    for (int e = 0; e < kN; ++e) outv[e] = (ea * inv) * outv[e] + (ec * inv) * oc[e];
    lse2 = mx + __log2f(ea + ec);
  }
  __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(P.out) + (size_t)hq * kD + d;
  if constexpr (kN == 4) *reinterpret_cast<uint2*>(out) = make_uint2(pack_bf16(outv[0], outv[1]), pack_bf16(outv[2], outv[3]));
  else *out = __float2bfloat16_rn(outv[0]);
  if (d == 0) {
    if (P.lse_out) P.lse_out[hq] = lse2 * kLn2;
    if (P.flags)
      P.flags[hq] = (uint8_t)((apply ? 1 : 0) | (rho < a.theta1 ? 2 : 0) | (a.n_cal <= 64 ? (cs << 2) : 0));
  }
}
__device__ __forceinline__ void merge_store(const DecodeCommon& a, const DecodeLayerPtrs& P, int hq, int d, float acc,
                                            float M, float Lsum, unsigned long long best, float lse_c, float oc) {
  const float acc1[1] = {acc}, oc1[1] = {oc};
  merge_store<1>(a, P, hq, d, acc1, M, Lsum, best, lse_c, oc1);
}

// Algorithm 2, lines 4-6, for the launches that recompute a calibration entry: the attention of the
// current query over the (reloaded) evicted KV is the new O_c row, its log-denominator the new LSE_c,
// and the query itself the new C_q row (the reading of line 4-5's "Q_-1" as the current query).
__device__ __forceinline__ void recal_store(const DecodeCommon& a, const DecodeLayerPtrs& P, int hq, int d, float acc,
                                            float M, float Lsum) {
  const size_t row = (size_t)hq * a.n_cal + a.recal_slot;
  const_cast<float*>(P.O_c)[row * kD + d] = acc / Lsum;
  reinterpret_cast<__nv_bfloat16*>(const_cast<void*>(P.C_q))[row * kD + d] =
      reinterpret_cast<const __nv_bfloat16*>(P.q)[(size_t)hq * kD + d];
  if (d == 0) const_cast<float*>(P.LSE_c)[row] = (M + log2f(Lsum)) * kLn2;
}

// RECAL = false: the decode step.  RECAL = true: the same stream over the evicted KV, without the
// similarity and the gate, ending in recal_store.  S: the shape of a CTA.
template <int NL, bool RECAL, class S>
__global__ void __launch_bounds__(S::kThreads, S::kCtas)
decode_kernel(const __grid_constant__ DecodeArgsT<NL> args) {
  constexpr int kSlots = S::kSlots, kSlotRows = S::kRows, kSubs = S::kSubs, kStreamWarps = S::kStreamWarps;
  constexpr int kThreads = S::kThreads, kPlaneBytes = S::kPlaneBytes, kSlotBytes = S::kSlotBytes;
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long s_full[kSlots][2], s_empty[kSlots][2];
  __shared__ unsigned long long s_best[kMaxG];     // best (similarity, row) of this CTA's calibration rows
  __shared__ unsigned long long s_bestall[kMaxG];  // ... of the whole cluster
  __shared__ __align__(8) unsigned long long s_bestx[S::kClu][kMaxG];   // ... of every CTA, pushed by them
  __shared__ __align__(8) unsigned long long s_bestbar;
  __shared__ __align__(16) float s_xpart[kMaxG * kD];  // [source split][head][dim of this CTA's slice]
  __shared__ __align__(16) float s_xml[S::kClu][kMaxG][2];   // [source split][head] (max, sum)
  __shared__ __align__(8) unsigned long long s_push;  // counts the bytes pushed to this CTA by the cluster
  __shared__ __align__(16) uint4 s_q[S::kClu == 1 && !RECAL ? kMaxG * kD / 8 : 1];  // the unit's queries
  __shared__ __align__(8) unsigned long long s_qfull;
  __shared__ int s_abort;
  __shared__ unsigned s_ticket;

  const DecodeCommon& a = args.c;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // ---- (0) overlap with the kernel ahead of this one in the stream, first thing in the kernel: an
  // L2 prefetch of the head of this CTA's slice of the retained cache.  Until the dependency wait
  // nothing the predecessor may have written is read and nothing global is written; a prefetch
  // cannot observe stale data (L2 is the point of coherence) and turns the head of the later TMA
  // stream into L2 hits.  Only the head: about what HBM delivers until the dependency wait is
  // released.  A deeper prefetch queues so much in the memory system that the small, latency-
  // critical loads of q and C_q behind it come back late (measured: 3/8 of the slice is best).
  if (threadIdx.x == kStreamWarps * 32) {
    const int pr0 = min(a.n_kv, (int)blockIdx.x * a.rows_per_split);
    const int pr1 = min(a.n_kv, pr0 + a.rows_per_split);
    const int n_old = min(min(pr1, a.kv_len) - pr0, (3 * a.rows_per_split + 7) / 8);
    if (n_old > 0) {
      const uint64_t pol = policy_evict_first();
      const size_t off = ((size_t)blockIdx.y * a.cap + pr0) * kRowBytes;
      const unsigned bytes = (unsigned)n_old * kRowBytes;
      asm volatile("cp.async.bulk.prefetch.L2.global.L2::cache_hint [%0], %1, %2;" ::"l"(
                       (const unsigned char*)args.layer[blockIdx.z].K + off),
                   "r"(bytes), "l"(pol)
                   : "memory");
      asm volatile("cp.async.bulk.prefetch.L2.global.L2::cache_hint [%0], %1, %2;" ::"l"(
                       (const unsigned char*)args.layer[blockIdx.z].V + off),
                   "r"(bytes), "l"(pol)
                   : "memory");
    }
  }
  cg::cluster_group cluster = cg::this_cluster();
  constexpr bool kOne = S::kClu == 1;    // a unit is one CTA's: nothing to combine across CTAs
  const int nsplit = kOne ? 1 : a.nsplit, nclu = kOne ? 1 : a.nclu;
  const int gs = kOne ? 0 : blockIdx.x;  // split index over the whole unit
  const int split = gs % nsplit;         // rank inside the cluster
  const int clu = gs / nsplit;           // cluster of this unit
  const int n_gs = nsplit * nclu;
  const int unit = blockIdx.y, layer = blockIdx.z;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int gq = lane >> 2, tq = lane & 3;  // MMA fragment coordinates
  const DecodeLayerPtrs& P = args.layer[layer];
  const DecodeLayerMaps& TM = args.maps[layer];
  const int b = unit / a.Hkv, h = unit % a.Hkv;
  const int hq0 = b * a.Hq + h * a.G;  // first query head of this kv group

  const __nv_bfloat16* q = (const __nv_bfloat16*)P.q;
  const __nv_bfloat16* Cq = (const __nv_bfloat16*)P.C_q;

  const int r0 = min(a.n_kv, gs * a.rows_per_split);
  const int r1 = min(a.n_kv, r0 + a.rows_per_split);
  // Ring fills of this CTA: the K/V rows, and with one CTA per unit the unit's calibration queries ahead of them, 32 rows
  // per warp of the slot.
  constexpr int kCalRows = kSubs * 32;
  const int n_cf = kOne && !RECAL ? (a.G * a.n_cal + kCalRows - 1) / kCalRows : 0;
  const int n_sb = n_cf + (r1 - r0 + kSlotRows - 1) / kSlotRows;

  const uint64_t pol_stream = policy_evict_first(), pol_keep = policy_evict_last();
  const uint32_t ring = (smem_u32(smem_raw) + 1023u) & ~1023u;
  unsigned char* ring_ptr = smem_raw + (ring - smem_u32(smem_raw));
  volatile int* abort_flag = &s_abort;

  // calibration rows of this CTA: the contiguous range [c_begin, c_begin + n_c)
  const int c_per = (a.n_cal + n_gs - 1) / n_gs;
  const int c_begin = min(a.n_cal, gs * c_per);
  const int n_c = RECAL ? 0 : min(a.n_cal, c_begin + c_per) - c_begin;
  if (tid == 0) {
    for (int s = 0; s < kSlots; ++s)
      for (int p = 0; p < 2; ++p) {
        if (s == 0 && p == 0) mbar_init(smem_u32(&s_qfull), 1);
        mbar_init(smem_u32(&s_full[s][p]), 1);    // the producer's arrive with the byte count
        mbar_init(smem_u32(&s_empty[s][p]), kSubs);   // one lane of each of the slot's warps
      }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_abort = 0;
  }
  if (warp == kStreamWarps && lane == 0) {
    // every CTA of the cluster (this one included) pushes its partial of this CTA's slice and its
    // (max, sum) pairs here: G * dpc * 4 + G * 8 bytes each
    mbar_init(smem_u32(&s_push), 1);
    mbar_init(smem_u32(&s_bestbar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (!kOne) mbar_expect_tx(smem_u32(&s_push), (uint32_t)(nsplit * a.G * (kD / nsplit * 4 + 8)));
    if (!kOne && !RECAL) mbar_expect_tx(smem_u32(&s_bestbar), (uint32_t)(nsplit * a.G * 8));
    asm volatile("prefetch.tensormap [%0];" ::"l"(&TM.k64) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&TM.v64) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&TM.k16) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&TM.v16) : "memory");
  }
  if (tid >= 32 && tid < 32 + a.G && n_c > 0) {  // same for the small operands of the similarity
    const int g = tid - 32;
    asm volatile("cp.async.bulk.prefetch.L2.global.L2::cache_hint [%0], %1, %2;" ::"l"(
                     Cq + ((size_t)(hq0 + g) * a.n_cal + c_begin) * kD),
                 "r"((unsigned)n_c * kRowBytes), "l"(pol_keep)
                 : "memory");
    if (g == 0)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(q + (size_t)hq0 * kD),
                   "r"((unsigned)a.G * kRowBytes)
                   : "memory");
  }
  if (tid < kMaxG) s_best[tid] = 0ull;
  // Address arithmetic of everything that is loaded right after the dependency wait, and of the
  // finish, is done here: a single warp runs a dependent chain of scalar instructions at a few
  // cycles each, and at this kernel's scale a hundred of them behind the wait are a measurable
  // part of a launch (0.4 us each for the similarity loads and for the O_c loads, measured).
  // (the stream warps': the producer has the first fills to send off)
  constexpr int kPairsPerPass = kStreamWarps * 8;
  const int pairs = warp == kStreamWarps ? 0 : n_c * a.G;
  const int sub4 = tid & 3;
  const int pi0 = tid >> 2;
  const int pg0 = pi0 < pairs ? pi0 % a.G : 0, pc0 = c_begin + (pi0 < pairs ? pi0 / a.G : 0);
  const uint4* qp0 = reinterpret_cast<const uint4*>(q + (size_t)(hq0 + pg0) * kD + sub4 * 32);
  const uint4* cp0 = reinterpret_cast<const uint4*>(Cq + ((size_t)(hq0 + pg0) * a.n_cal + pc0) * kD + sub4 * 32);
  const uint32_t* qr0 = reinterpret_cast<const uint32_t*>(q + (size_t)(hq0 + min(gq, a.G - 1)) * kD) + tq;
  const int dpc = kD / nsplit, lg_dpc = 31 - __clz(dpc);  // nsplit is a power of two
  const int n_items = a.G * dpc;
  const bool single = nclu == 1;
  // threads that share an output element in the finish, each with up to four splits: as many as there are threads for
  const int lg_sub = nsplit >= 4 && n_items * 4 <= kThreads ? 2 : nsplit >= 2 && n_items * 2 <= kThreads ? 1 : 0;
  const bool early = !kOne && !RECAL && single && n_items << lg_sub <= kThreads;  // one output element per thread at most
  const int eg = min(tid >> lg_sub >> lg_dpc, a.G - 1), ed = split * dpc + ((tid >> lg_sub) & (dpc - 1));
  const float* oc_base = P.O_c + (size_t)(hq0 + eg) * a.n_cal * kD + ed;
  const float* lsec_base = P.LSE_c + (size_t)(hq0 + eg) * a.n_cal;
  asm volatile("" ::"l"(qp0), "l"(cp0), "l"(qr0), "l"(oc_base), "l"(lsec_base), "r"(pg0), "r"(pc0));
  __syncthreads();  // barriers initialised, s_best cleared: nothing of this needs the predecessor
  // (A) arrived at once, waited for ahead of a warp's first push: every CTA of the cluster runs, its barriers are set up
  if (!kOne) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");

  // One ring fill into slot sb % kSlots: calibration queries first where they go through the ring, then kSlotRows rows of
  // K and V.  Whole slots of 64 rows take a 64-row box each, or one for each half of the columns; slots of 32 rows and the ragged
  // last one take 16-row boxes for the row groups that hold valid rows.  Slices begin at multiples of 16 rows, so none of these
  // brings rows of a neighbour, and the results rely on that (a probability of zero times an infinite value of V is NaN).  Only a
  // 16-row box can reach past row kv_len: the V map of those boxes ends at kv_len, so such V rows arrive as zeros (a zero
  // probability times whatever lies in the caller's memory could still be a NaN); the K rows
  // arrive as they lie in memory and their scores are masked.
  auto fill = [&](int sb) {
    const int s = sb % kSlots, k = sb / kSlots;
    const uint32_t bar = smem_u32(&s_full[s][k & 1]);
    const uint32_t dst = ring + s * kSlotBytes;
    if (kOne && sb < n_cf) {
      const int rows = min(kCalRows, a.G * a.n_cal - sb * kCalRows);
      const unsigned bytes = (unsigned)rows * kRowBytes, q_bytes = (unsigned)a.G * kRowBytes;
      if (sb == 0) {
        mbar_expect_tx(smem_u32(&s_qfull), q_bytes);
        bulk_load(smem_u32(s_q), q + (size_t)hq0 * kD, q_bytes, smem_u32(&s_qfull), pol_keep);
      }
      mbar_expect_tx(bar, bytes);
      bulk_load(dst, Cq + ((size_t)hq0 * a.n_cal + sb * kCalRows) * kD, bytes, bar, pol_keep);
      return;
    }
    const int row0 = r0 + (sb - n_cf) * kSlotRows;
    const int nrows = min(kSlotRows, r1 - row0);
    if (kSlotRows == kWideRows && nrows == kSlotRows) {
      mbar_expect_tx(bar, kSlotBytes);
      const bool halves = RECAL ? a.half_copies != 0 : S::kHalf;   // (see DecodeCommon)
      tma_load_rows(dst, &TM.k64, bar, row0, unit, pol_stream);
      if (halves) tma_load_rows(dst + kPlaneBytes, &TM.k64, bar, row0, unit, pol_stream, 1);
      tma_load_rows(dst + 2 * kPlaneBytes, &TM.v64, bar, row0, unit, pol_stream);
      if (halves) tma_load_rows(dst + 3 * kPlaneBytes, &TM.v64, bar, row0, unit, pol_stream, 1);
    } else {
      const int nb = (nrows + kBlkRows - 1) / kBlkRows;
      mbar_expect_tx(bar, (uint32_t)nb * 4u * kBlkRows * 128u);
      for (int j = 0; j < nb; ++j) {
        const uint32_t dj = dst + j * 2 * kBlkRows * 128;
        tma_load_rows(dj, &TM.k16, bar, row0 + j * kBlkRows, unit, pol_stream);
        tma_load_rows(dj + 2 * kPlaneBytes, &TM.v16, bar, row0 + j * kBlkRows, unit, pol_stream);
      }
    }
  };

  // ---- (1) cosine similarities of this CTA's calibration rows: four lanes per (head, row) pair,
  // kPairsPerPass pairs per pass; the best pair per head goes to s_best while the first slots are in flight
  auto rho_load = [&](int pi, RhoLoad (&r)[2]) {
    r[0] = RhoLoad{}; r[1] = RhoLoad{};
    if (pi < pairs) {
      const int g = pi % a.G, c = c_begin + pi / a.G;
      const uint4* qp = reinterpret_cast<const uint4*>(q + (size_t)(hq0 + g) * kD + sub4 * 32);
      const uint4* cp = reinterpret_cast<const uint4*>(Cq + ((size_t)(hq0 + g) * a.n_cal + c) * kD + sub4 * 32);
      r[0].q0 = __ldg(qp); r[0].q1 = __ldg(qp + 1);
      r[0].c0 = ldg_keep(cp, pol_keep); r[0].c1 = ldg_keep(cp + 1, pol_keep);
      r[1].q0 = __ldg(qp + 2); r[1].q1 = __ldg(qp + 3);
      r[1].c0 = ldg_keep(cp + 2, pol_keep); r[1].c1 = ldg_keep(cp + 3, pol_keep);
    }
  };
  auto rho_finish = [&](int pi, int g, int c, const RhoLoad (&r)[2]) {
    float dot = 0.f, qq = 0.f, cc = 0.f;
    if (pi < pairs) { rho_accumulate(r[0], dot, qq, cc); rho_accumulate(r[1], dot, qq, cc); }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
      dot += __shfl_xor_sync(0xffffffffu, dot, o);
      qq += __shfl_xor_sync(0xffffffffu, qq, o);
      cc += __shfl_xor_sync(0xffffffffu, cc, o);
    }
    if (sub4 == 0 && pi < pairs) {
      const float rho = (qq > 0.f && cc > 0.f) ? dot / (sqrtf(qq) * sqrtf(cc)) : 0.f;
      atomicMax(&s_best[g], rank_key(rho, c));
    }
  };
  // query fragments of the stream warps (B operand of S^T, heads on the 8-column side): their
  // loads go out together with those of the similarity
  uint32_t qa[kD / 16][2];
#pragma unroll
  for (int kk = 0; kk < kD / 16; ++kk) {
    qa[kk][0] = 0u; qa[kk][1] = 0u;
    if (warp < kStreamWarps && gq < a.G) {
      qa[kk][0] = __ldg(qr0 + kk * 8);
      qa[kk][1] = __ldg(qr0 + kk * 8 + 4);
    }
  }
  RhoLoad rl[2];
  rl[0] = RhoLoad{}; rl[1] = RhoLoad{};
  if (!kOne && pi0 < pairs) {
    rl[0].q0 = __ldg(qp0); rl[0].q1 = __ldg(qp0 + 1);
    rl[0].c0 = ldg_keep(cp0, pol_keep); rl[0].c1 = ldg_keep(cp0 + 1, pol_keep);
    rl[1].q0 = __ldg(qp0 + 2); rl[1].q1 = __ldg(qp0 + 3);
    rl[1].c0 = ldg_keep(cp0 + 2, pol_keep); rl[1].c1 = ldg_keep(cp0 + 3, pol_keep);
  }
  // the first ring fills go out behind the (small) similarity loads, not ahead of them
  if (warp == kStreamWarps) {
    if (lane == 0)
      for (int sb = 0; sb < min(n_sb, kSlots); ++sb) fill(sb);
    __syncwarp();
  }
  // A stream warp finishes its similarities after its first slot, whose data is already there when the query arrives.  The stream
  // warps then hand their updates of s_best to the producer warp through a CTA barrier, and that one, which has no similarities and
  // time, pushes them to the CTAs of the cluster.
  auto rho_rest = [&]() {
    if (kOne) return;
    rho_finish(pi0, pg0, pc0, rl);
    for (int base = kPairsPerPass; base < pairs; base += kPairsPerPass) {
      const int pi = base + pi0;
      rho_load(pi, rl);
      rho_finish(pi, pi < pairs ? pi % a.G : 0, c_begin + (pi < pairs ? pi / a.G : 0), rl);
    }
    if (warp != kStreamWarps) asm volatile("barrier.cta.arrive 1, %0;" ::"n"(kThreads) : "memory");
  };
  // One CTA per unit: the similarities of a slot of calibration queries, a row per lane.  (Loaded through registers, four
  // lanes to a row, the passes were a chain of round trips that held the stream up: 73 instead of 60 us for 2048 caches
  // of 231 rows.)
  // The sums are those of the other shapes, to the bit, so that no near-tie between two rows depends on the shape: quarters
  // of a row, each in ascending order, added in pairs.  (Every second group of four lanes takes a pair's quarters the other way
  // round, which halves the bank conflicts; lanes that start up to three chunks apart and meet in no bank were slower,
  // 63.5 us.)
  auto rho_slot = [&](int s, int sb, int sub) {
    const int rows = a.G * a.n_cal, r = sb * kCalRows + sub * 32 + lane;
    const int g_lo = (sb * kCalRows + sub * 32) / a.n_cal, g = r < rows ? r / a.n_cal : -1, c = r - g * a.n_cal;
    if (g_lo >= a.G) return;                          // (the same for the whole warp)
    const uint4* crow = reinterpret_cast<const uint4*>(ring_ptr + s * kSlotBytes) + (sub * 32 + lane) * (kD / 8);
    const uint4* qrow = s_q + (g < 0 ? 0 : g) * (kD / 8);
    float dot = 0.f, qq = 0.f, cc = 0.f;
    const int parity = (lane >> 2) & 1;
#pragma unroll 1
    for (int pair = 0; pair < 2; ++pair) {
      float d[2] = {0.f, 0.f}, dq[2] = {0.f, 0.f}, dc[2] = {0.f, 0.f};
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int chunk = (2 * pair + (e ^ parity)) * 4;
#pragma unroll
        for (int j = 0; j < 4; ++j) rho_accumulate(qrow[chunk + j], crow[chunk + j], d[e], dq[e], dc[e]);
      }
      dot += d[0] + d[1]; qq += dq[0] + dq[1]; cc += dc[0] + dc[1];
    }
    const float rho = (qq > 0.f && cc > 0.f) ? dot / (sqrtf(qq) * sqrtf(cc)) : 0.f;
    const unsigned hi = (unsigned)(rank_key(rho, 0) >> 32);
    const int g_hi = min(a.G - 1, (sb * kCalRows + sub * 32 + 31) / a.n_cal);
    for (int gg = g_lo; gg <= g_hi; ++gg) {
      const unsigned m = __reduce_max_sync(0xffffffffu, g == gg ? hi : 0u);
      const unsigned cm = __reduce_max_sync(0xffffffffu, g == gg && hi == m ? (unsigned)c : 0u);
      if (lane == 0) atomicMax(&s_best[gg], ((unsigned long long)m << 32) | cm);
    }
  };

  float o[kD / 16][4];
#pragma unroll
  for (int n = 0; n < kD / 16; ++n) { o[n][0] = o[n][1] = o[n][2] = o[n][3] = 0.f; }
  float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;  // heads 2tq and 2tq+1

  if (warp == kStreamWarps) {
    rho_rest();
    // ---- (2) producer: refill a slot as soon as its four warps have released it
    if (lane == 0) {
      for (int sb = kSlots; sb < n_sb; ++sb) {
        const int s = sb % kSlots, kp = sb / kSlots - 1;  // the fill that occupies the slot
        if (!mbar_wait(smem_u32(&s_empty[s][kp & 1]), (kp >> 1) & 1, abort_flag, a.status, 0x100u + sb)) break;
        fill(sb);
      }
    }
    __syncwarp();
    // with the last fill under way the producer has nothing left to move: it settles the
    // calibration row (best similarity over the cluster, ties to the largest row index) while the
    // stream warps are still busy
    if (!kOne) asm volatile("barrier.cta.sync 1, %0;" ::"n"(kThreads) : "memory");  // the stream warps' updates of s_best
    if (!kOne) cluster_wait();   // (A)
    if (!kOne && !RECAL) {
      // Pushed like the partial outputs below.  (Published by a release of the whole CTA at a cluster barrier and read from
      // the peers, this took a microsecond of fence while copies are in flight and a chain of remote loads: 8 units of 129
      // rows 4.96 -> 4.5 us a launch, longer streams cover it.)
      if ((lane & 7) < a.G) {
        const unsigned long long mine = s_best[lane & 7];
#pragma unroll
        for (int r0 = 0; r0 < S::kClu; r0 += 4) {
          const int r = r0 + (lane >> 3);
          if (r < nsplit)
            push_u64(cluster_addr(smem_u32(&s_bestx[split][lane & 7]), r), mine, cluster_addr(smem_u32(&s_bestbar), r));
        }
      }
      mbar_wait_sit_out(smem_u32(&s_bestbar), 0, abort_flag, a.status, 0x500u);
      if (lane < a.G) {
        unsigned long long best = 0ull;
#pragma unroll
        for (int s = 0; s < S::kClu; ++s) {
          const unsigned long long k = s < nsplit ? s_bestx[s][lane] : 0ull;
          best = k > best ? k : best;
        }
        s_bestall[lane] = best;
      }
    }
  } else {
    // ---- (3) stream warps
    const int group = warp / kSubs, sub = warp % kSubs;
    const int mid = lane >> 3;
    bool rho_done = false;
    for (int sb = group; sb < n_sb; sb += 2) {
      const int s = sb % kSlots, k = sb / kSlots;
      const int row_base = r0 + (sb - n_cf) * kSlotRows + sub * kBlkRows;
      // D1: the warp that meets row kv_len takes it from k_new / v_new, on their way while the slot is.  (Loaded once the slot had
      // arrived, 8 units x 700 rows took 4.89 instead of 4.71 us.  Rows of calibration queries have a row_base of -16 at most.)
      const bool new_row = !RECAL && a.has_new && a.kv_len >= row_base && a.kv_len < row_base + kBlkRows;
      uint4 v_new;
      if (new_row)
        v_new = *reinterpret_cast<const uint4*>((const unsigned char*)(lane < 16 ? P.k_new : P.v_new) +
                                                (size_t)unit * kRowBytes + (lane & 15) * 16);
      const bool ok = mbar_wait(smem_u32(&s_full[s][k & 1]), (k >> 1) & 1, abort_flag, a.status, 0x200u + sb);
      if (kOne && sb < n_cf) {
        if (!RECAL && ok && mbar_wait(smem_u32(&s_qfull), 0, abort_flag, a.status, 0x400u)) rho_slot(s, sb, sub);
      } else if (ok && row_base < r1) {
        const Planes pl = planes_of<S>(kSlotRows == kWideRows && r1 - r0 - (sb - n_cf) * kSlotRows >= kSlotRows);
        const uint32_t sK = ring + s * kSlotBytes + sub * pl.block;   // this warp's block
        const uint32_t sV = sK + 2 * kPlaneBytes;
        // ... and appends it to the cache (whose row has not been written yet: what arrived for it is stale)
        if (new_row) {
          const int chunk = lane & 15;
          const int rs = a.kv_len - row_base;  // row inside the block
          unsigned char* dstg = (unsigned char*)(lane < 16 ? P.K : P.V) +
                                ((size_t)unit * a.cap + a.kv_len) * kRowBytes + chunk * 16;
          *reinterpret_cast<uint4*>(dstg) = v_new;
          *reinterpret_cast<uint4*>(ring_ptr + s * kSlotBytes + sub * pl.block + (lane < 16 ? 0 : 2 * kPlaneBytes) +
                                    block_off(pl, rs, chunk)) = v_new;
          __syncwarp();
        }
        // S^T: two accumulators (even and odd k-steps) halve the dependent chain
        float sa[4] = {0.f, 0.f, 0.f, 0.f}, sb2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int kk = 0; kk < kD / 16; ++kk) {
          uint32_t a0, a1, a2, a3;
          ldmatrix_x4(sK + block_off(pl, (lane & 7) + (mid & 1) * 8, kk * 2 + (mid >> 1)), a0, a1, a2, a3);
          if (kk & 1) mma_bf16_16816(sb2, a0, a1, a2, a3, qa[kk][0], qa[kk][1]);
          else mma_bf16_16816(sa, a0, a1, a2, a3, qa[kk][0], qa[kk][1]);
        }
        // online softmax per head over the 16 keys of the block (keys gq and gq + 8 live here)
        const bool v0 = row_base + gq < r1, v1 = row_base + gq + 8 < r1;
        const float x00 = v0 ? (sa[0] + sb2[0]) * a.scale2 : -INFINITY;
        const float x01 = v0 ? (sa[1] + sb2[1]) * a.scale2 : -INFINITY;
        const float x10 = v1 ? (sa[2] + sb2[2]) * a.scale2 : -INFINITY;
        const float x11 = v1 ? (sa[3] + sb2[3]) * a.scale2 : -INFINITY;
        float bm0 = fmaxf(x00, x10), bm1 = fmaxf(x01, x11);
#pragma unroll
        for (int off = 4; off < 32; off <<= 1) {
          bm0 = fmaxf(bm0, __shfl_xor_sync(0xffffffffu, bm0, off));
          bm1 = fmaxf(bm1, __shfl_xor_sync(0xffffffffu, bm1, off));
        }
        const float mn0 = fmaxf(m0, bm0), mn1 = fmaxf(m1, bm1);  // finite: the block's first key is valid
        const float corr0 = ex2_approx(m0 - mn0), corr1 = ex2_approx(m1 - mn1);
        const float p00 = ex2_approx(x00 - mn0), p01 = ex2_approx(x01 - mn1);
        const float p10 = ex2_approx(x10 - mn0), p11 = ex2_approx(x11 - mn1);
        l0 = l0 * corr0 + (p00 + p10);  // partial over this thread's keys, summed over gq at the end
        l1 = l1 * corr1 + (p01 + p11);
        m0 = mn0; m1 = mn1;
#pragma unroll
        for (int n = 0; n < kD / 16; ++n) { o[n][0] *= corr0; o[n][1] *= corr1; o[n][2] *= corr0; o[n][3] *= corr1; }
        // P^T as the B operand: transpose the two 8x8 (key, head) fragments inside the warp
        const uint32_t pb0 = movmatrix_trans(pack_bf16(p00, p01)), pb1 = movmatrix_trans(pack_bf16(p10, p11));
#pragma unroll
        for (int n = 0; n < kD / 16; ++n) {
          uint32_t a0, a1, a2, a3;
          ldmatrix_x4_trans(sV + block_off(pl, (lane & 7) + (mid >> 1) * 8, n * 2 + (mid & 1)), a0, a1, a2, a3);
          mma_bf16_16816(o[n], a0, a1, a2, a3, pb0, pb1);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&s_empty[s][k & 1]));  // the slot may be refilled
      if (!rho_done) { rho_rest(); rho_done = true; }
    }
    if (!rho_done) rho_rest();
#pragma unroll
    for (int off = 4; off < 32; off <<= 1) {
      l0 += __shfl_xor_sync(0xffffffffu, l0, off);
      l1 += __shfl_xor_sync(0xffffffffu, l1, off);
    }
  }

  // ---- (4) the chosen O_c elements and LSE_c start their way while the partials are combined
  if (!kOne && warp < kStreamWarps) cluster_wait();  // (A)
  __syncthreads();  // all warps are done with the ring: reuse it for the combine
  // the common case has one output element per thread at most: its O_c element and LSE_c are
  // loaded now and arrive while the partials are combined
  if (!kOne && !RECAL && (!single || n_items > kThreads)) {
    if (tid < a.G && single) {
      const size_t crow = (size_t)(hq0 + tid) * a.n_cal + (unsigned)(s_bestall[tid] & 0xffffffffull);
      const float* orow = P.O_c + crow * kD;
#pragma unroll
      for (int i = 0; i < 4; ++i) asm volatile("prefetch.global.L2 [%0];" ::"l"(orow + i * 32));
      asm volatile("prefetch.global.L2 [%0];" ::"l"(P.LSE_c + crow));
    }
  }
  float lse_c_early = 0.f, oc_early = 0.f;
  if (early && tid < n_items << lg_sub) {
    const unsigned cs = (unsigned)(s_bestall[eg] & 0xffffffffull);
    lse_c_early = ldg_keep(lsec_base + cs, pol_keep);
    oc_early = ldg_keep(oc_base + (size_t)cs * kD, pol_keep);
  }

  // one CTA per unit: a warp per head, four elements per thread, the first head's O_c on its way now
  uint4 oc_one = make_uint4(0u, 0u, 0u, 0u);
  auto load_oc = [&](int g) {
    const size_t crow = (size_t)(hq0 + g) * a.n_cal + (unsigned)(s_best[g] & 0xffffffffull);
    oc_one = ldg_keep(reinterpret_cast<const uint4*>(P.O_c + crow * kD) + lane, pol_keep);
    lse_c_early = ldg_keep(P.LSE_c + crow, pol_keep);
  };
  if (kOne && !RECAL && warp < min(kStreamWarps, a.G)) load_oc(warp);

  // ---- (5) CTA combine of the stream warps, pushed to the owners of the output slices:
  // CTA r of the cluster owns dimensions [r * dpc, (r + 1) * dpc) of every head of the group
  float* wo = reinterpret_cast<float*>(ring_ptr);          // [warp][8][kWoStride]
  float* wml = wo + kStreamWarps * kMaxG * kWoStride;       // [warp][8][2]
  if (warp < kStreamWarps && 2 * tq < a.G) {
#pragma unroll
    for (int n = 0; n < kD / 16; ++n) {
      float* w0 = wo + (warp * kMaxG + 2 * tq) * kWoStride + n * 16 + gq;
      w0[0] = o[n][0]; w0[8] = o[n][2];
      w0[kWoStride] = o[n][1]; w0[kWoStride + 8] = o[n][3];
    }
    if (gq == 0) {
      wml[(warp * kMaxG + 2 * tq) * 2] = m0; wml[(warp * kMaxG + 2 * tq) * 2 + 1] = l0;
      wml[(warp * kMaxG + 2 * tq + 1) * 2] = m1; wml[(warp * kMaxG + 2 * tq + 1) * 2 + 1] = l1;
    }
  }
  __syncthreads();
  if constexpr (kOne) {
    if (warp < kStreamWarps) {
      for (int g = warp; g < a.G; g += kStreamWarps) {
        if (!RECAL && g != warp) load_oc(g);
        float mw[kStreamWarps], M = -INFINITY, Lsum = 0.f, acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int w = 0; w < kStreamWarps; ++w) { mw[w] = wml[(w * kMaxG + g) * 2]; M = fmaxf(M, mw[w]); }
#pragma unroll
        for (int w = 0; w < kStreamWarps; ++w) {
          const float sc = mw[w] > -INFINITY ? ex2_approx(mw[w] - M) : 0.f;
          const float4 v = *reinterpret_cast<const float4*>(wo + (w * kMaxG + g) * kWoStride + 4 * lane);
          Lsum = fmaf(wml[(w * kMaxG + g) * 2 + 1], sc, Lsum);
          acc[0] = fmaf(v.x, sc, acc[0]); acc[1] = fmaf(v.y, sc, acc[1]);
          acc[2] = fmaf(v.z, sc, acc[2]); acc[3] = fmaf(v.w, sc, acc[3]);
        }
        if constexpr (RECAL) {
          for (int e = 0; e < 4; ++e) recal_store(a, P, hq0 + g, 4 * lane + e, acc[e], M, Lsum);
        } else {
          const float oc[4] = {__uint_as_float(oc_one.x), __uint_as_float(oc_one.y), __uint_as_float(oc_one.z),
                               __uint_as_float(oc_one.w)};
          merge_store<4>(a, P, hq0 + g, 4 * lane, acc, M, Lsum, s_best[g], lse_c_early, oc);
        }
      }
    }
    return;
  }
  // A warp per head, four elements a lane: the scale factors of the stream warps are worked out once for four elements,
  // which go to their owner in one 16-byte store; all loads are done before the pushes (stores through generic pointers,
  // which the compiler will not move loads across).
  if (warp < min(kStreamWarps, a.G)) {
    const int g = warp, d0 = 4 * lane;
    float mw[kStreamWarps], M = -INFINITY, Lsum = 0.f;
#pragma unroll
    for (int w = 0; w < kStreamWarps; ++w) { mw[w] = wml[(w * kMaxG + g) * 2]; M = fmaxf(M, mw[w]); }
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int w = 0; w < kStreamWarps; ++w) {
      const float sc = mw[w] > -INFINITY ? ex2_approx(mw[w] - M) : 0.f;
      const float4 v = *reinterpret_cast<const float4*>(wo + (w * kMaxG + g) * kWoStride + d0);
      Lsum = fmaf(wml[(w * kMaxG + g) * 2 + 1], sc, Lsum);
      acc.x = fmaf(v.x, sc, acc.x); acc.y = fmaf(v.y, sc, acc.y);
      acc.z = fmaf(v.z, sc, acc.z); acc.w = fmaf(v.w, sc, acc.w);
    }
    const int own = d0 >> lg_dpc;  // dpc is a multiple of eight: the four dimensions have the same owner
    push_f32x4(cluster_addr(smem_u32(s_xpart + (split * kMaxG + g) * dpc + (d0 - own * dpc)), own), acc,
               cluster_addr(smem_u32(&s_push), own));
    if (lane < nsplit)  // the (max, sum) pair of this split goes to every CTA of the cluster
      push_f32x2(cluster_addr(smem_u32(&s_xml[split][g][0]), lane), M, Lsum, cluster_addr(smem_u32(&s_push), lane));
  }
  // (B) everything pushed to this CTA has arrived when its byte count is complete.  No cluster
  // barrier: a CTA waits for its own data only, and nothing else of a peer touches its shared memory.
  // The wait has to be sat out: a CTA whose earlier wait ran out (abort flag raised) must not skip it,
  // or its peers, which always reach their pushes, would write to the shared memory of a
  // CTA that has left.  Only the wait's own time limit remains as the way out.
  mbar_wait_sit_out(smem_u32(&s_push), 0, abort_flag, a.status, 0x300u);

  // ---- (6) finish: reduce the splits for this CTA's output slice (local data only from here on,
  // so no CTA has to wait for another before it leaves)
  // A split after another in one thread, the sixteen of a cluster took 2200 cycles, most of them for fetching 250 instructions
  // that run once per launch; with four threads to an element it is a quarter of the code and of the chain.
  const int lu = layer * a.units + unit;
  constexpr int kMine = 4;   // splits of a thread at most: elements get fewer threads only where there are few splits
  const int sub = tid & ((1 << lg_sub) - 1);
  for (int item = tid >> lg_sub; item < n_items; item += kThreads >> lg_sub) {   // (a warp's items are in range all or none)
    const int g = item >> lg_dpc, dl = item & (dpc - 1), d = split * dpc + dl;
    const int hq = hq0 + g;
    const unsigned long long best = s_bestall[g];
    float ms[kMine], ls[kMine], xs[kMine], M = -INFINITY;
#pragma unroll
    for (int k = 0; k < kMine; ++k) {  // all loads first
      const int s = (k << lg_sub) + sub;
      const bool on = s < nsplit;
      ms[k] = on ? s_xml[s][g][0] : -INFINITY;
      ls[k] = on ? s_xml[s][g][1] : 0.f;
      xs[k] = on ? s_xpart[(s * kMaxG + g) * dpc + dl] : 0.f;
      M = fmaxf(M, ms[k]);
    }
    if (lg_sub > 0) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, 1));
    if (lg_sub > 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, 2));
    float Lsum = 0.f, acc = 0.f;
#pragma unroll
    for (int k = 0; k < kMine; ++k) {
      const float sc = ms[k] > -INFINITY ? ex2_approx(ms[k] - M) : 0.f;
      Lsum = fmaf(ls[k], sc, Lsum);
      acc = fmaf(xs[k], sc, acc);
    }
    if (lg_sub > 0) { Lsum += __shfl_xor_sync(0xffffffffu, Lsum, 1); acc += __shfl_xor_sync(0xffffffffu, acc, 1); }
    if (lg_sub > 1) { Lsum += __shfl_xor_sync(0xffffffffu, Lsum, 2); acc += __shfl_xor_sync(0xffffffffu, acc, 2); }
    if (sub != 0) continue;
    if (single) {
      if constexpr (RECAL) {
        recal_store(a, P, hq, d, acc, M, Lsum);
      } else {
        float lse_c = lse_c_early, oc = oc_early;
        if (!early) {
          const size_t crow = (size_t)hq * a.n_cal + (unsigned)(best & 0xffffffffull);
          lse_c = __ldg(P.LSE_c + crow);
          oc = __ldg(P.O_c + crow * kD + d);
        }
        merge_store(a, P, hq, d, acc, M, Lsum, best, lse_c, oc);
      }
    } else {
      // this cluster's partial goes to the workspace; (M, Lsum, best) are the same in all its CTAs
      const size_t pc = ((size_t)lu * nclu + clu) * kMaxG + g;
      a.part_o[pc * kD + d] = acc;
      if (d == 0) {
        a.part_ml[pc * 2] = M;
        a.part_ml[pc * 2 + 1] = Lsum;
        a.part_best[pc] = best;
      }
    }
  }
  if (!single) {
    // ---- (7) several clusters per unit: the CTA that takes the unit's last ticket merges them
    __threadfence();
    __syncthreads();
    if (tid == 0) s_ticket = atomicAdd(&a.counters[lu], 1u);
    __syncthreads();
    if (s_ticket == (unsigned)(n_gs - 1)) {
      __threadfence();
      for (int gd = tid; gd < a.G * kD; gd += kThreads) {
        const int g = gd / kD, d = gd % kD;
        const size_t pu = (size_t)lu * nclu * kMaxG + g;
        unsigned long long best = 0ull;
        float ms[8], ls[8], os[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          ms[c] = -INFINITY; ls[c] = 0.f; os[c] = 0.f;
          if (c < nclu) {
            const size_t pc = pu + (size_t)c * kMaxG;
            const unsigned long long k = __ldcg(a.part_best + pc);
            best = k > best ? k : best;
            const float2 ml2 = __ldcg(reinterpret_cast<const float2*>(a.part_ml + pc * 2));
            ms[c] = ml2.x; ls[c] = ml2.y;
            os[c] = __ldcg(a.part_o + pc * kD + d);
          }
        }
        const int hq = hq0 + g;
        const size_t crow = (size_t)hq * a.n_cal + (unsigned)(best & 0xffffffffull);
        const float lse_c = RECAL ? 0.f : __ldg(P.LSE_c + crow);
        const float oc = RECAL ? 0.f : __ldg(P.O_c + crow * kD + d);
        float M = -INFINITY;
#pragma unroll
        for (int c = 0; c < 8; ++c) M = fmaxf(M, ms[c]);
        float Lsum = 0.f, acc = 0.f;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const float sc = ms[c] > -INFINITY ? ex2_approx(ms[c] - M) : 0.f;
          Lsum = fmaf(ls[c], sc, Lsum);
          acc = fmaf(os[c], sc, acc);
        }
        if constexpr (RECAL) recal_store(a, P, hq, d, acc, M, Lsum);
        else merge_store(a, P, hq, d, acc, M, Lsum, best, lse_c, oc);
      }
      if (tid == 0) a.counters[lu] = 0u;  // ready for the next launch on this workspace
    }
  }
}

}  // namespace

bool make_decode_maps(const DecodeCommon& c, const DecodeLayerPtrs& L, DecodeLayerMaps* out) {
  // Three of the four maps cover all `cap` rows of the cache, whatever kv_len is, so one encoding
  // serves every step on a cache: a small per-thread table keyed by everything the encoding depends
  // on (the two base addresses, the capacity, the number of units, the kind of copies) returns them on the following
  // calls (encoding all four on every call cost more host time than the kernel runs).  An entry can
  // never be stale: equal keys encode equal maps.  The fourth, V in 16-row boxes, is the only one
  // through which rows at or beyond kv_len can reach a product; it ends at kv_len, so the TMA unit
  // delivers zeros for those rows, and is encoded per call.
  struct Entry { const void* K; const void* V; int cap, units, half_copies; DecodeLayerMaps maps; };
  constexpr int kEntries = 64;
  static thread_local Entry table[kEntries];
  static thread_local int next = 0;
  const uint64_t strides[2] = {(uint64_t)kRowBytes, (uint64_t)c.cap * kRowBytes};
  const uint32_t box64[2] = {(uint32_t)kWideRows, 1}, box16[2] = {(uint32_t)kBlkRows, 1};
  const uint64_t dims_v16[2] = {(uint64_t)(c.kv_len > 0 ? c.kv_len : 1), (uint64_t)c.units};
  for (int i = 0; i < kEntries; ++i) {
    const Entry& e = table[i];
    if (e.K == L.K && e.V == L.V && e.cap == c.cap && e.units == c.units && e.half_copies == c.half_copies && e.K != nullptr) {
      *out = e.maps;
      return make_tile_map_bf16(&out->v16, L.V, 3, dims_v16, strides, box16, 2);
    }
  }
  const uint64_t dims[2] = {(uint64_t)c.cap, (uint64_t)c.units};
  const int halves = c.half_copies ? 1 : 2;
  if (!(make_tile_map_bf16(&out->k64, L.K, 3, dims, strides, box64, halves) &&
        make_tile_map_bf16(&out->v64, L.V, 3, dims, strides, box64, halves) &&
        make_tile_map_bf16(&out->k16, L.K, 3, dims, strides, box16, 2) &&
        make_tile_map_bf16(&out->v16, L.V, 3, dims_v16, strides, box16, 2)))
    return false;
  Entry& e = table[next];
  next = (next + 1) % kEntries;
  e.K = L.K; e.V = L.V; e.cap = c.cap; e.units = c.units; e.half_copies = c.half_copies; e.maps = *out;
  return true;
}

namespace {

template <int NL, bool RECAL, class S>
cudaError_t setup_decode(int dev) {
  static std::atomic<bool> done[64];
  if (dev >= 0 && dev < 64 && done[dev].load(std::memory_order_acquire)) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(decode_kernel<NL, RECAL, S>, cudaFuncAttributeMaxDynamicSharedMemorySize, S::kSmemBytes);
  if (e == cudaSuccess && S::kClu > 8)
    e = cudaFuncSetAttribute(decode_kernel<NL, RECAL, S>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev].store(true, std::memory_order_release);
  return e;
}

template <int NL, bool RECAL, class S>
cudaError_t launch_decode_s(const DecodeArgsT<NL>& a, cudaStream_t st) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = setup_decode<NL, RECAL, S>(dev);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(a.c.nsplit * a.c.nclu, a.c.units, a.c.n_layers);
  cfg.blockDim = dim3(S::kThreads);
  cfg.dynamicSmemBytes = S::kSmemBytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;  // the splits of a unit are one cluster
  attr[0].val.clusterDim.x = a.c.nsplit;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  e = cudaLaunchKernelEx(&cfg, decode_kernel<NL, RECAL, S>, a);
  if (e != cudaSuccess) return e;
  count_launch(1);
  return cudaGetLastError();
}

// More units than SMs (a stack of caches in one launch), a CTA each: smaller rings, fewer warps and the calibration queries
// through the ring, so that several CTAs share an SM and one's fixed chain overlaps the others' streams.  Two CTAs per SM
// as long as that is all of them, else four.  Against the wide ring, one CTA per SM (us): 256 caches of 2049 rows 56.8 ->
// 48.9, 192 of 800 28.6 -> 20.1, 1024 of 1000 122 -> 107, 512 of 800 62 -> 46.5; 704 of 1300 equal and 384 of 2000 75 -> 80: long
// slices of more CTAs than fit two to an SM keep it.  2048 of 231 rows: two CTAs of eight stream warps with the similarities
// through registers 88.9, four of four warps 73, with the calibration queries through the ring 60 (48 for the bytes).
constexpr int kNarrowRows = 1024;

template <int NL, bool RECAL, bool kHalf>
cudaError_t launch_decode_h(const DecodeArgsT<NL>& a, cudaStream_t st) {
  switch (decode_ctas_per_sm(a.c)) {
    case 4: return launch_decode_s<NL, RECAL, ShapeNarrow>(a, st);
    case 2: return launch_decode_s<NL, RECAL, ShapePair<kHalf>>(a, st);
  }
  if constexpr (!RECAL)
    if (a.c.nsplit > 8) return launch_decode_s<NL, RECAL, ShapeCluster16<kHalf>>(a, st);
  return launch_decode_s<NL, RECAL, ShapeWide<kHalf>>(a, st);
}

template <int NL, bool RECAL>
cudaError_t launch_decode_t(const DecodeArgsT<NL>& a, cudaStream_t st) {
  if constexpr (!RECAL)
    if (a.c.half_copies) return launch_decode_h<NL, RECAL, true>(a, st);
  return launch_decode_h<NL, RECAL, false>(a, st);
}

}  // namespace

int decode_ctas_per_sm(const DecodeCommon& c) {
  const long long ctas = (long long)c.nsplit * c.nclu * c.units * c.n_layers;
  if (ctas > 2 * kDecodeTargetCtas && c.rows_per_split <= kNarrowRows) return 4;
  return ctas > kDecodeTargetCtas && ctas <= 2 * kDecodeTargetCtas ? 2 : 1;
}

cudaError_t launch_decode(const DecodeArgsT<1>& a, cudaStream_t st) { return launch_decode_t<1, false>(a, st); }
cudaError_t launch_decode(const DecodeArgsT<kDecodeMaxLayers>& a, cudaStream_t st) {
  return launch_decode_t<kDecodeMaxLayers, false>(a, st);
}
int decode_resident_clusters(int ctas) {
  static std::atomic<int> known[64][5];   // per device and log2 of the size; 0: not asked yet, else 1 + clusters
  int dev = 0, lg = 0;
  while ((1 << lg) < ctas) ++lg;
  if (lg > 4 || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  int n = known[dev][lg].load(std::memory_order_acquire);
  if (n == 0) {
    // (the kernels of one shape differ in their arguments only)
    int active = 0;
    if (setup_decode<1, false, ShapeCluster16<false>>(dev) != cudaSuccess) return 0;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(ShapeCluster16<false>::kThreads);
    cfg.dynamicSmemBytes = ShapeCluster16<false>::kSmemBytes;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = ctas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&active, decode_kernel<1, false, ShapeCluster16<false>>, &cfg) != cudaSuccess) {
      cudaGetLastError();   // no such cluster on this device
      active = 0;
    }
    n = 1 + active;
    known[dev][lg].store(n, std::memory_order_release);
  }
  return n - 1;
}
cudaError_t launch_recalibrate(const DecodeArgsT<1>& a, cudaStream_t st) { return launch_decode_t<1, true>(a, st); }

}  // namespace calidrop
