// Pooling + per-(batch, kv-head) top-k on thread-block clusters.
//
// A cluster of 1..16 CTAs shares a unit: CTA r owns the contiguous key range [r * chunk, (r + 1) * chunk),
// every thread keeps its ROWS keys (pooled votes as fp32 bit patterns; non-negative, so unsigned order is
// numeric order) in registers, and the CTAs exchange only histograms and counts through distributed
// shared memory.  Exact radix select, digits of 8 + 8 + 8 + 7 bits (the sign bit is zero), finds a threshold
// T and how many candidates equal to T are taken besides all those above it; an ordered compaction then
// emits them ascending (ties go to the lowest index), plus the kept bitmap.  With a calibration size
// the second threshold is searched in the same passes.
//
// What bounds it is latency: barriers and the round trips between them; no pipe or memory is near a limit.
// Hence
//   * the votes are staged in shared memory once, with the pool's halo, instead of `pool` loads per key;
//   * votes have few exponents, so the first digits fall into a handful of bins: a histogram has a column
//     per LANE (word bin * 32 + lane), so that the lanes of a warp never meet in a word or a bank;
//   * three barriers per pass: the columns of a bin are summed by one warp reduction and cleared as they
//     are read, the sums are PUSHED to every CTA of the cluster, and one warp per threshold walks them;
//   * the passes end as soon as all keys of the chosen bin are taken (usually after two or three);
//   * key (warp w, row i, lane l) of CTA r is candidate r * chunk + (w * ROWS + i) * 32 + l: a warp owns a
//     contiguous run, so the compaction scans one count per warp (a ballot is one bitmap word);
//   * the cluster is only as large as the prompt needs: a prompt of 2048 keys takes one CTA and no
//     cluster barrier at all.
// Measured, kernel time from cold caches, against 1024-thread clusters of eight with a histogram per warp,
// pooled from global memory: 64 units x 16384 keys 33.3 -> 18.8 us, 32 x 32768 24.8 -> 20.6 us, 4 x 131072 36.8 -> 29.4 us,
// 16 x 5003 with a calibration size 22.8 -> 19.2 us, 8 x 8192 11.9 -> 13.8 us (in a stream of calls, beside the
// neighbouring kernels, 1.2 us less per call all the same).  Wider digits, 11 + 10 + 10 bits with two
// histograms per CTA, were slower, 47 us at 32 x 32768: the votes' few exponents share bins.
// Then, the partial votes loaded in batches (they were a chain of round trips) and sixteen CTAs for a unit where few
// units share the GPU: compress calls of 4 x 131072 keys 339 -> 325 us, 32 x 32768 379 -> 371 us, 64 x 16384 184 -> 180 us.
#include <cooperative_groups.h>

#include <atomic>
#include <type_traits>

#include "common.cuh"
#include "internal.h"

namespace calidrop {

namespace {

namespace cg = cooperative_groups;

constexpr int kPortableClu = 8, kMaxClu = 16;   // clusters of more than eight CTAs where few units leave the GPU idle
constexpr int kHaloMax = 64;   // widest half pool that is staged; wider pools read the votes from global memory

struct SelectArgs {
  const float* votes;     // [part][unit][stride]: the partial votes (or the caller's scores, one part)
  float* vote_sum;        // out [units, n_cand]: the summed votes, or null
  float* pooled;          // out [units, n_cand]
  uint32_t* bitmap;       // out [units, bitmap_words]
  uint32_t* mask2;        // out, kSized: bit set = not one of the calibrated evicted rows
  int32_t* kept_idx;      // out [units, n_kept]
  size_t stride, part_stride;
  int n_parts, n_cand, L, pool, k_sel, n_kept, bitmap_words, n_calib;
};

// kClu: the most CTAs a cluster of this instantiation has.
template <int T, int ROWS, bool kSized, int kClu>
__global__ void __launch_bounds__(T)
pool_select_cluster_kernel(const SelectArgs a) {
  constexpr int kW = T / 32;
  constexpr int kChunk = ROWS * T;
  constexpr int kThr = kSized ? 2 : 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned* const hist = reinterpret_cast<unsigned*>(smem_raw);            // [kThr][256][32]
  unsigned* const counts = hist + kThr * 256 * 32;   // [2][kThr][kClu][256]: every CTA's histogram (double-buffered)
  float* const stage = reinterpret_cast<float*>(counts + 2 * kThr * kClu * 256);   // [kChunk + 2 * kHaloMax]
  auto counts_of = [&](int buf, int x, int r) { return counts + ((buf * kThr + x) * kClu + r) * 256; };
  __shared__ unsigned sel_bin[kThr], sel_k[kThr], sel_all[kThr];
  __shared__ unsigned cnt[kClu][kThr][2];         // every CTA's keys > T and == T, per threshold
  __shared__ unsigned wcnt[kThr][32][2];          // this CTA's, per warp

  pdl_trigger();
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), n_clu = (int)cluster.num_blocks();
  const int unit = blockIdx.y;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < kThr * 256 * 8; i += T) reinterpret_cast<uint4*>(hist)[i] = make_uint4(0u, 0u, 0u, 0u);
  const int c0 = rank * kChunk;
  const int n_cand = a.n_cand;
  const int half = a.pool >> 1;
  const float* v = a.votes + (size_t)unit * a.stride;
  float* pl = a.pooled + (size_t)unit * n_cand;
  uint32_t* bm = a.bitmap + (size_t)unit * a.bitmap_words;
  int32_t* kept = a.kept_idx + (size_t)unit * a.n_kept;
  const float fpool = (float)a.pool;
  // (a CTA may store into a peer's shared memory only once the peer runs: waited for ahead of the first push)
  if (n_clu > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  pdl_wait();

  // 1. zero-padded average pool with a constant divisor; keys stay in registers
  auto vote_at = [&](int t) {
    float x = v[t];
    for (int p = 1; p < a.n_parts; ++p) x += v[(size_t)p * a.part_stride + t];
    return x;
  };
  const bool staged = half <= kHaloMax;
  if (staged) {
    const int n_stage = min(kChunk, n_cand - c0) + 2 * half;   // (not positive when only window rows are left)
    float* const vs = a.vote_sum ? a.vote_sum + (size_t)unit * n_cand : nullptr;
    // up to 16 loads of a thread in flight: one position after the other, a thread of a 131072-key prompt walked 64
    // dependent round trips here (4 parts of 16 keys: 30.5 of 75 thousand cycles)
    auto stage_parts = [&](auto parts_tag) __attribute__((always_inline)) {
      constexpr int kParts = decltype(parts_tag)::value;
      constexpr int kBatch = ROWS < 16 / kParts ? ROWS : 16 / kParts;
#pragma unroll 1
      for (int i0 = tid; i0 < n_stage; i0 += kBatch * T) {
        float x[kBatch][kParts];
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
          const int i = i0 + j * T, t = c0 - half + i;
          const bool in = i < n_stage && t >= 0 && t < n_cand;
#pragma unroll
          for (int q = 0; q < kParts; ++q) x[j][q] = in ? __ldcg(v + (size_t)q * a.part_stride + t) : 0.f;
        }
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
          const int i = i0 + j * T, own = i - half;
          float sum = x[j][0];
#pragma unroll
          for (int q = 1; q < kParts; ++q) sum += x[j][q];
          if (i < n_stage) {
            stage[i] = sum;
            if (vs && own >= 0 && own < min(kChunk, n_cand - c0)) vs[c0 + own] = sum;
          }
        }
      }
    };
    if (a.n_parts == 1) stage_parts(std::integral_constant<int, 1>{});
    else if (a.n_parts == 2) stage_parts(std::integral_constant<int, 2>{});
    else stage_parts(std::integral_constant<int, 4>{});
  }
  __syncthreads();
  unsigned key[ROWS];
  auto pooled_key = [&](int t, float acc) {
    const float p = acc / fpool;
    pl[t] = p;
    return (unsigned)max(__float_as_int(p), 0);   // (a score below zero or a negative NaN ranks as zero)
  };
  auto pool_rows = [&](auto taps_tag) __attribute__((always_inline)) {
    constexpr int kTaps = decltype(taps_tag)::value;
#pragma unroll
    for (int i = 0; i < ROWS; ++i) {
      const int tl = (warp * ROWS + i) * 32 + lane, t = c0 + tl;
      key[i] = 0u;
      if (t < n_cand) {
        float acc = 0.f;
#pragma unroll
        for (int d = 0; d < kTaps; ++d) acc += stage[tl + d];
        key[i] = pooled_key(t, acc);
      }
    }
  };
  switch (a.pool) {
    case 1: pool_rows(std::integral_constant<int, 1>{}); break;
    case 5: pool_rows(std::integral_constant<int, 5>{}); break;
    case 7: pool_rows(std::integral_constant<int, 7>{}); break;
    default:
#pragma unroll
      for (int i = 0; i < ROWS; ++i) {
        const int tl = (warp * ROWS + i) * 32 + lane, t = c0 + tl;
        key[i] = 0u;
        if (t < n_cand) {
          float acc = 0.f;
          for (int d = -half; d <= half; ++d) {
            if (staged) acc += stage[tl + half + d];
            else if (t + d >= 0 && t + d < n_cand) acc += vote_at(t + d);
          }
          key[i] = pooled_key(t, acc);
        }
      }
  }
  if (a.vote_sum && !staged)
    for (int i = tid; i < min(kChunk, n_cand - c0); i += T)
      a.vote_sum[(size_t)unit * n_cand + c0 + i] = vote_at(c0 + i);
  if (n_clu > 1) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");

  // 2. radix select, most significant digit first.  thr[x] ends as the threshold of selection x, k[x] as the
  // number of keys equal to it that are taken.
  unsigned prefix[kThr], k[kThr], thr[kThr];
  bool open[kThr];
#pragma unroll
  for (int x = 0; x < kThr; ++x) {
    prefix[x] = 0u; thr[x] = 0u; open[x] = true;
    k[x] = (unsigned)(a.k_sel + (x ? a.n_calib : 0));
  }
#pragma unroll 1
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = pass == 3 ? 0 : 23 - 8 * pass, bits = pass == 3 ? 7 : 8;
#pragma unroll
    for (int i = 0; i < ROWS; ++i) {
      const bool valid = c0 + (warp * ROWS + i) * 32 + lane < n_cand;
#pragma unroll
      for (int x = 0; x < kThr; ++x)
        if (valid && open[x] && (key[i] >> shift >> bits) == prefix[x])   // (pass 0: the sign bit, zero)
          atomicAdd(hist + (x * 256 + ((key[i] >> shift) & ((1u << bits) - 1u))) * 32 + lane, 1u);
    }
    __syncthreads();
    constexpr int kPer = 256 / kW;   // bins of a warp
#pragma unroll
    for (int x = 0; x < kThr; ++x) {
      unsigned m = 0u;
#pragma unroll
      for (int j = 0; j < kPer; ++j) {
        unsigned* h = hist + (x * 256 + warp * kPer + j) * 32 + lane;
        const unsigned s = __reduce_add_sync(0xffffffffu, *h);
        *h = 0u;
        if (lane == j) m = s;
      }
      // pushed to every CTA of the cluster: stores to a peer cost no round trip, loads from it would
      if (lane < kPer)
        for (int r = 0; r < n_clu; ++r)
          cluster.map_shared_rank(counts_of(pass & 1, x, rank), r)[warp * kPer + lane] = m;
    }
    if (n_clu > 1) cluster.sync();
    else __syncthreads();
    // one warp per threshold: lane 0 owns the 8 highest bins; walk downwards until k keys are covered
    if (warp < kThr) {
      const int x = warp;
      unsigned c[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
#pragma unroll
      for (int r = 0; r < kClu; ++r) {
        const uint4* h = reinterpret_cast<const uint4*>(counts_of(pass & 1, x, r)) + 2 * (31 - lane);
        uint4 lo = make_uint4(0u, 0u, 0u, 0u), hi = lo;
        if (r < n_clu) { lo = h[0]; hi = h[1]; }
        c[7] += lo.x; c[6] += lo.y; c[5] += lo.z; c[4] += lo.w;
        c[3] += hi.x; c[2] += hi.y; c[1] += hi.z; c[0] += hi.w;
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
    __syncthreads();
    bool any = false;
#pragma unroll
    for (int x = 0; x < kThr; ++x) {
      if (!open[x]) continue;
      prefix[x] = (prefix[x] << bits) | sel_bin[x];
      thr[x] = prefix[x] << shift;
      k[x] = sel_k[x];
      // every key of the bin is taken: so is every key at or above the bin's lowest bit pattern
      if (sel_all[x]) { k[x] = 0xffffffffu; open[x] = false; }
      any |= open[x];
    }
    if (!any) break;
  }

  // 3. ordered compaction.  Number of keys above / equal to a threshold in the warps and CTAs ahead of this warp.
  unsigned before_gt[kThr], before_eq[kThr];
#pragma unroll
  for (int x = 0; x < kThr; ++x) {
    unsigned g = 0u, e = 0u;
#pragma unroll
    for (int i = 0; i < ROWS; ++i) {
      const bool valid = c0 + (warp * ROWS + i) * 32 + lane < n_cand;
      g += __popc(__ballot_sync(0xffffffffu, valid && key[i] > thr[x]));
      e += __popc(__ballot_sync(0xffffffffu, valid && key[i] == thr[x]));
    }
    if (lane == 0) { wcnt[x][warp][0] = g; wcnt[x][warp][1] = e; }
  }
  __syncthreads();
#pragma unroll
  for (int x = 0; x < kThr; ++x) {
    const unsigned g = lane < kW ? wcnt[x][lane][0] : 0u, e = lane < kW ? wcnt[x][lane][1] : 0u;
    before_gt[x] = __reduce_add_sync(0xffffffffu, lane < warp ? g : 0u);
    before_eq[x] = __reduce_add_sync(0xffffffffu, lane < warp ? e : 0u);
    if (n_clu > 1 && warp == 0) {
      const unsigned sg = __reduce_add_sync(0xffffffffu, g), se = __reduce_add_sync(0xffffffffu, e);
      if (lane < n_clu) {
        unsigned* c = cluster.map_shared_rank(&cnt[rank][x][0], lane);
        c[0] = sg; c[1] = se;
      }
    }
  }
  if (n_clu > 1) {
    // the last time a CTA touches a peer's shared memory lies ahead of this barrier: it may leave afterwards
    cluster.sync();
#pragma unroll
    for (int x = 0; x < kThr; ++x) {
      before_gt[x] += __reduce_add_sync(0xffffffffu, lane < rank ? cnt[lane][x][0] : 0u);
      before_eq[x] += __reduce_add_sync(0xffffffffu, lane < rank ? cnt[lane][x][1] : 0u);
    }
  }
  const unsigned lt = (1u << lane) - 1u;
#pragma unroll
  for (int i = 0; i < ROWS; ++i) {
    const int t0 = c0 + (warp * ROWS + i) * 32, t = t0 + lane;
    const bool valid = t < n_cand;
    const unsigned gm = __ballot_sync(0xffffffffu, valid && key[i] > thr[0]);
    const unsigned em = __ballot_sync(0xffffffffu, valid && key[i] == thr[0]);
    const unsigned gt_before = before_gt[0] + __popc(gm & lt), eq_before = before_eq[0] + __popc(em & lt);
    before_gt[0] += __popc(gm);
    before_eq[0] += __popc(em);
    // (observation-window rows are always kept)
    const bool sel = valid && (key[i] > thr[0] || (key[i] == thr[0] && eq_before < k[0]));
    if (sel) kept[gt_before + min(eq_before, k[0])] = t;
    const bool take = sel || (!valid && t < a.L);
    const unsigned word = __ballot_sync(0xffffffffu, take);
    if (lane == 0 && t0 < a.L) bm[t0 >> 5] = word;
    if (kSized) {
      // calibration size: the candidates among the first k_sel + n_calib that were not selected
      constexpr int y = kThr - 1;
      const unsigned em2 = __ballot_sync(0xffffffffu, valid && key[i] == thr[y]);
      const bool in2 = valid && (key[i] > thr[y] || (key[i] == thr[y] && before_eq[y] + __popc(em2 & lt) < k[y]));
      before_eq[y] += __popc(em2);
      const unsigned word2 = ~__ballot_sync(0xffffffffu, in2 && !take);
      if (lane == 0 && t0 < a.L) a.mask2[(size_t)unit * a.bitmap_words + (t0 >> 5)] = word2;
    }
  }
  // the window rows close the kept list
  if (rank == 0)
    for (int j = tid; j < a.L - n_cand; j += T) kept[a.k_sel + j] = n_cand + j;
}

template <int T, int ROWS, bool kSized, int kClu>
struct Launch {
  static constexpr int kSmem = ((kSized ? 2 : 1) * (256 * 32 + 2 * kClu * 256) + ROWS * T + 2 * kHaloMax) * 4;

  static void config(int n_clu, int units, cudaStream_t st, cudaLaunchConfig_t& cfg, cudaLaunchAttribute (&attr)[2]) {
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3(n_clu, units);
    cfg.blockDim = dim3(T);
    cfg.dynamicSmemBytes = kSmem;
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

  // What the current device needs set up once.  `resident`: clusters of kClu CTAs it runs at the same time (only asked
  // for beyond the portable size, where the shape of the device's processor clusters decides).
  static cudaError_t setup(int* resident) {
    static std::atomic<int> known[64];   // 0: not set up yet, else 1 + resident
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool slot = dev >= 0 && dev < 64;
    int n = slot ? known[dev].load(std::memory_order_acquire) : 0;
    if (n == 0) {
      auto* kernel = pool_select_cluster_kernel<T, ROWS, kSized, kClu>;
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
      if (e != cudaSuccess) return e;
      int active = 0;
      if (kClu > kPortableClu) {
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr[2];
        config(kClu, 1, nullptr, cfg, attr);
        cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&active, kernel, &cfg) != cudaSuccess) {
          cudaGetLastError();   // no such cluster on this device
          active = 0;
        }
      }
      n = 1 + active;
      if (slot) known[dev].store(n, std::memory_order_release);
    }
    if (resident) *resident = n - 1;
    return cudaSuccess;
  }

  static bool all_resident(const SelectArgs& a, int units) {
    int resident = 0;
    return a.L <= kClu * T * ROWS && setup(&resident) == cudaSuccess && units <= resident;
  }

  static cudaError_t run(const SelectArgs& a, int units, cudaStream_t st) {
    cudaError_t e = setup(nullptr);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    config((a.L + T * ROWS - 1) / (T * ROWS), units, st, cfg, attr);
    e = cudaLaunchKernelEx(&cfg, pool_select_cluster_kernel<T, ROWS, kSized, kClu>, a);
    count_launch(1);
    return e != cudaSuccess ? e : cudaGetLastError();
  }
};

template <bool kSized>
cudaError_t launch_any(const SelectArgs& a, int units, cudaStream_t st) {
  // The fewest keys per thread with which all clusters of the call are resident at once, two CTAs of 512
  // threads per SM: the work per thread is what a pass waits for (1024-thread CTAs with 16 keys per thread:
  // 32 units x 32768 keys 29.0 us instead of 20.6, 64 x 16384 25.2 instead of 18.8), but clusters beyond a
  // full GPU would queue.  Below 2048 keys per CTA nothing is gained (1024 threads with one or two keys: equal).
  auto clusters = [&](int chunk) { return (a.L + chunk - 1) / chunk; };
  auto fits = [&](int rows) {
    const int c = clusters(512 * rows);
    return c <= kPortableClu && (long long)c * units <= 2 * kSms;
  };
  if (fits(4)) return Launch<512, 4, kSized, kPortableClu>::run(a, units, st);
  if (fits(8)) return Launch<512, 8, kSized, kPortableClu>::run(a, units, st);
  // Longer prompts of few units: up to sixteen CTAs per unit, half the keys per thread.
  if (a.L > kPortableClu * 512 * 8) {
    using C8 = Launch<1024, 8, kSized, kMaxClu>;
    using C16 = Launch<1024, 16, kSized, kMaxClu>;
    if (C8::all_resident(a, units)) return C8::run(a, units, st);
    if (a.L > kPortableClu * 1024 * 16 && C16::all_resident(a, units)) return C16::run(a, units, st);
  }
  if (a.L <= kPortableClu * 512 * 16) return Launch<512, 16, kSized, kPortableClu>::run(a, units, st);
  if (a.L <= kPortableClu * 1024 * 16) return Launch<1024, 16, kSized, kPortableClu>::run(a, units, st);
  return Launch<1024, 32, kSized, kPortableClu>::run(a, units, st);
}

}  // namespace

// The cluster kernel keeps at most 32 keys per thread: 8 CTAs x 1024 threads x 32.
bool select_cluster_supported(const CompressGeom& g) { return !g.keep_all && g.L <= kPortableClu * 1024 * 32; }

// Selection from per-candidate scores [parts][units][stride] (the window votes of the workspace, or a
// caller's scores); vote_sum receives the sum of the parts when it is not null.
cudaError_t launch_pool_select_scores(const CompressGeom& g, const CompressWs& ws, char* wsp, const float* scores,
                                      size_t stride, int n_parts, size_t part_stride, float* vote_sum,
                                      int32_t* kept_idx, cudaStream_t st) {
  SelectArgs a{};
  a.votes = scores;
  a.vote_sum = vote_sum;
  a.pooled = (float*)(wsp + ws.pooled);
  a.bitmap = (uint32_t*)(wsp + ws.bitmap);
  a.kept_idx = kept_idx;
  a.stride = stride; a.part_stride = part_stride; a.n_parts = n_parts;
  a.n_cand = g.n_cand; a.L = g.L; a.pool = g.pool; a.k_sel = g.k_sel; a.n_kept = g.n_kept;
  a.bitmap_words = g.bitmap_words;
  if (g.sized && g.n_calib > 0) {
    a.mask2 = (uint32_t*)(wsp + ws.bitmap2);
    a.n_calib = g.n_calib;
    return launch_any<true>(a, g.units, st);
  }
  return launch_any<false>(a, g.units, st);
}

// Selection from the window votes of the workspace: ws.vote, or with `in_parts` the partial votes that
// launch_votes_tc left, whose sum goes to ws.vote on the way.
cudaError_t launch_pool_select_cluster(const CompressGeom& g, const CompressWs& ws, char* wsp, bool in_parts,
                                       int32_t* kept_idx, cudaStream_t st) {
  float* vote = (float*)(wsp + ws.vote);
  if (!in_parts) return launch_pool_select_scores(g, ws, wsp, vote, (size_t)g.n_cand, 1, 0, nullptr, kept_idx, st);
  return launch_pool_select_scores(g, ws, wsp, (const float*)(wsp + ws.vote_parts), (size_t)g.n_cand, votes_tc_parts(g),
                                   (size_t)g.units * g.n_cand, vote, kept_idx, st);
}

// Sink-plus-recent index rule: the first n_sink rows and the last n_kept - n_sink.
__global__ void streaming_indices_kernel(int32_t* __restrict__ kept_idx, int L, int n_kept, int n_sink) {
  const int unit = blockIdx.y, i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n_kept) kept_idx[(size_t)unit * n_kept + i] = i < n_sink ? i : L - (n_kept - i);
}

cudaError_t launch_streaming_indices(const CompressGeom& g, int n_sink, int32_t* kept_idx, cudaStream_t st) {
  streaming_indices_kernel<<<dim3((g.n_kept + 255) / 256, g.units), 256, 0, st>>>(kept_idx, g.L, g.n_kept, n_sink);
  count_launch(1);
  return cudaGetLastError();
}

}  // namespace calidrop
