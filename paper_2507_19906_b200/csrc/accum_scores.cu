// Accumulated attention scores of a prompt, the importance measure of the H2O eviction rule
// (Sections 4.1.2-4.1.3 apply the calibration on top of it): for every (batch, kv head) and every
// key t, the causal softmax attention that key receives, summed over the prompt's queries i >= t and
// over the query heads of the group.  Serving code gets these sums as a by-product of the prefill
// attention; this file computes them from Q and K for callers that have none, in two passes on the
// tensor cores (tcgen05, bf16 products, fp32 logits, statistics and sums):
//   pass 1  row statistics: lse2[b, hq, i] = log2 sum_{t <= i} exp2(s2[i, t]),  s2 = q.k * scale * log2(e)
//   pass 2  column sums:    part[b, hq, t] = sum_{i >= t} exp2(s2[i, t] - lse2[i])
// and score[b, h, t] = sum over the heads of the group of part.  Every sum is taken in a fixed order (no
// atomics), so the result is reproducible bit for bit.  The cost is that of the prefill attention itself
// (L^2 D flop per head), which is why it is not part of the compress step.
//
// Both passes are one kernel.  An ITEM is a tile of 128 rows of one query head, queries in pass 1 and keys in
// pass 2, that stays in shared memory with its rows on the tensor-memory lanes; the tiles of 256 keys (queries)
// that it may see are streamed past it, one MMA accumulator of 256 columns (a JOB) each, so a row's sum is a
// per-thread sum over columns.  Items cost between one job and L / 256 of them: they are dealt to persistent CTAs
// in the order of their cost, forwards and backwards in turn, so that all CTAs end together.  Roles as in
// the window scoring: four consumer warpgroups in two pairs on alternate jobs, each group half of the columns, a TMA
// producer, an MMA-issuing warp.  What bounds it is the exponentials, one per visible logit and pass (see exp2.cuh).
// Measured at 32 query heads on 8 kv heads, 8192 tokens: 312 + 331 us (506 and 539 thousand cycles, the
// special-function unit 77 % and 70 % busy), against 1302 + 1313 us with 64 x 64 tiles on mma.sync.
#include <type_traits>

#include "exp2.cuh"
#include "internal.h"
#include "tc_common.cuh"

namespace calidrop {

namespace {

using namespace tc;

constexpr int kGroups = 4;
constexpr int kProducerWarp = kGroups * 4;
constexpr int kMmaWarp = kGroups * 4 + 1;
constexpr int kThreads = kGroups * 128 + 64;
constexpr int kRows = 128, kCols = 256;             // an item's rows, a job's columns
constexpr int kABytes = kRows * 256, kBBytes = kCols * 256;
constexpr int kStages = 2;
constexpr int kSmem = 2 * kABytes + kStages * kBBytes + 1024;

struct AccumArgs {
  int Hq, G, L;
  int heads;      // B * Hq
  int n_rt, n_ct; // row tiles and column tiles of a prompt
  int items;      // heads * n_rt
  float scale2;
  float* lse2;    // [heads, L]: pass 1 out, pass 2 in
  float* part;    // [heads, L]: pass 2 out
  unsigned* status;
};

// The n-th item of a CTA in the order of decreasing cost, dealt forwards and backwards in turn; false past the end.
template <bool kSums>
__device__ __forceinline__ bool item_at(const AccumArgs& a, int n, int& head, int& rt, int& ct0, int& n_jobs) {
  const int p = (int)gridDim.x, c = (int)blockIdx.x;
  const int idx = n * p + ((n & 1) ? p - 1 - c : c);
  if (idx >= a.items) return false;
  const int rank = idx / a.heads;
  head = idx - rank * a.heads;
  if (kSums) {          // keys: the first tiles are seen by the most queries
    rt = rank;
    ct0 = rt >> 1;
    n_jobs = a.n_ct - ct0;
  } else {              // queries: the last tiles see the most keys
    rt = a.n_rt - 1 - rank;
    ct0 = 0;
    n_jobs = (rt >> 1) + 1;
  }
  return true;
}

template <bool kSums>
__global__ void __launch_bounds__(kThreads, 1)
accum_tc_kernel(const __grid_constant__ CUtensorMap a_map, const __grid_constant__ CUtensorMap b_map, const AccumArgs a) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long bars[16];
  __shared__ uint32_t tmem_slot;
  __shared__ Ctl ctl;
  __shared__ float2 xs[2][kGroups - 1][kRows];                      // partials of groups 1..3, per item parity
  __shared__ __align__(16) float nlse2_s[kSums ? kGroups * 4 : 1][kSums ? 128 : 4];   // -lse2 of a warp's columns

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t a_base = smem_base, b_base = smem_base + 2 * kABytes;
  const uint32_t bar0 = smem_u32(bars);
  auto a_full = [&](int s) { return bar0 + 8u * s; };
  auto a_empty = [&](int s) { return bar0 + 8u * (2 + s); };
  auto b_full = [&](int s) { return bar0 + 8u * (4 + s); };
  auto b_empty = [&](int s) { return bar0 + 8u * (6 + s); };
  auto t_full = [&](int s) { return bar0 + 8u * (8 + s); };
  auto t_empty = [&](int s) { return bar0 + 8u * (10 + s); };
  auto x_full = [&](int s) { return bar0 + 8u * (12 + s); };
  auto x_empty = [&](int s) { return bar0 + 8u * (14 + s); };

  if (tid == 0) {
    ctl.abort = 0;
    ctl.status = a.status;
    for (int s = 0; s < 2; ++s) {
      mbar_init(a_full(s), 1); mbar_init(a_empty(s), 1);
      mbar_init(b_full(s), 1); mbar_init(b_empty(s), 1);
      mbar_init(t_full(s), 1); mbar_init(t_empty(s), 256);
      mbar_init(x_full(s), 128 * (kGroups - 1)); mbar_init(x_empty(s), 128);
    }
    fence_mbar_init();
  }
  if (warp == kMmaWarp) {
    tmem_alloc(smem_u32(&tmem_slot), 512);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = tmem_slot;
  pdl_wait();

  if (warp == kProducerWarp) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      tma_prefetch_desc(&a_map);
      tma_prefetch_desc(&b_map);
      int head, rt, ct0, n_jobs, s = 0;
      uint32_t s_ph = 0;
      bool ok = true;
      for (int n = 0; ok && item_at<kSums>(a, n, head, rt, ct0, n_jobs); ++n) {
        const int unit = head / a.G, as = n & 1;   // (B * Hq heads in groups of G: the kv unit)
        if (!mbar_wait(&ctl, a_empty(as), ((n >> 1) & 1) ^ 1, 50u)) break;
        mbar_arrive_expect_tx(a_full(as), kABytes);
        for (int half = 0; half < 2; ++half)
          tma_load_3d(a_base + as * kABytes + half * (kABytes / 2), &a_map, a_full(as), half * kHalfCols, rt * kRows,
                      kSums ? unit : head);
        for (int j = 0; j < n_jobs; ++j) {
          ok = mbar_wait(&ctl, b_empty(s), s_ph ^ 1, 51u);
          if (!ok) break;
          mbar_arrive_expect_tx(b_full(s), kBBytes);
          for (int half = 0; half < 2; ++half)
            tma_load_3d(b_base + s * kBBytes + half * (kBBytes / 2), &b_map, b_full(s), half * kHalfCols,
                        (ct0 + j) * kCols, kSums ? head : unit);
          if (++s == kStages) { s = 0; s_ph ^= 1u; }
        }
      }
    }
  } else if (__shfl_sync(0xffffffffu, warp, 0) == kMmaWarp) {
    // ------------------------------------------------------------ MMA issuer (the warp as a whole, one lane issues)
    const uint32_t idesc = umma_idesc(kRows, kCols, false, false);
    const uint64_t da0 = smem_desc_sw128(a_base, 16u, 1024u), db0 = smem_desc_sw128(b_base, 16u, 1024u);
    const bool leader = elect_one();
    int head, rt, ct0, n_jobs, s = 0, buf = 0;
    uint32_t s_ph = 0, t_ph = 0;
    bool ok = true;
    for (int n = 0; ok && item_at<kSums>(a, n, head, rt, ct0, n_jobs); ++n) {
      const int as = n & 1;
      ok = __all_sync(0xffffffffu, mbar_wait(&ctl, a_full(as), (n >> 1) & 1, 52u));
      const uint64_t ad = desc_advance(da0, (uint32_t)as * kABytes);
#pragma unroll 1
      for (int j = 0; j < n_jobs && ok; ++j) {
        ok = mbar_wait(&ctl, b_full(s), s_ph, 53u);
        ok = ok && mbar_wait(&ctl, t_empty(buf), t_ph ^ 1, 54u);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after_sync();
        const uint32_t d = tmem_base + (uint32_t)(buf * kCols);
        const uint64_t bd = desc_advance(db0, (uint32_t)s * kBBytes);
        if (leader) {
          umma_ss_imm<0>(d, ad, bd, idesc);
#pragma unroll
          for (int kk = 1; kk < kD / 16; ++kk)
            umma_ss_imm<1>(d, desc_advance(ad, kmajor_step_bytes(kABytes / 2, kk)),
                           desc_advance(bd, kmajor_step_bytes(kBBytes / 2, kk)), idesc);
          umma_commit(t_full(buf));
          umma_commit(b_empty(s));
          if (j == n_jobs - 1) umma_commit(a_empty(as));
        }
        __syncwarp();
        if (++s == kStages) { s = 0; s_ph ^= 1u; }
        buf ^= 1;
        if (buf == 0) t_ph ^= 1u;
      }
    }
  } else {
    // ------------------------------------------------------------ accumulator consumers (see score_tc.cu)
    const int grp = warp >> 2, row = tid & 127, pair = grp >> 1, half = grp & 1;
    const uint32_t taddr = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(pair * kCols + half * 128);
    const uint32_t bar_full = t_full(pair), bar_empty = t_empty(pair);
    const f32x2 sc = pack2(a.scale2);
    uint32_t ph = 0;
    bool ok = true;
    int head, rt, ct0, n_jobs, j0 = 0;   // j0: the CTA's job number of the item's first job; job j goes to pair j % 2
    // column sums: -lse2 of this warp's columns of the next own job, four per lane, loaded a job ahead
    float nl_next[4] = {0.f, 0.f, 0.f, 0.f};
    auto load_nl = [&](int hd, int ct) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int i = ct * kCols + half * 128 + q * 32 + lane;
        nl_next[q] = i < a.L ? -__ldcg(a.lse2 + (size_t)hd * a.L + i) : -INFINITY;
      }
    };
    bool have_nl = false;
    int n = 0;
    for (; item_at<kSums>(a, n, head, rt, ct0, n_jobs); ++n) {
      float2 ml = make_float2(-1e30f, 0.f);    // row statistics: running (max, sum)
      f32x2 acc0 = 0ull, acc1 = 0ull;          // column sums
      const int first = (pair ^ j0) & 1;
      int nan_at = -1;                         // column sums: the last query of this lane's whose statistics are NaN
#pragma unroll 1
      for (int j = first; j < n_jobs; j += 2) {
        if (kSums) {
          if (!have_nl) load_nl(head, ct0 + j);
          // A query whose statistics are NaN must reach the keys it sees and no others, but a masked logit of -inf does not
          // outweigh it: it is left out of the sums (fmaxf drops a NaN), and its position is kept until the item's end.
          __syncwarp();
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if (nl_next[q] != nl_next[q]) nan_at = (ct0 + j) * kCols + half * 128 + q * 32 + lane;
            nlse2_s[warp][q * 32 + lane] = fmaxf(nl_next[q], -INFINITY);
          }
          __syncwarp();
          have_nl = j + 2 < n_jobs;
          if (have_nl) load_nl(head, ct0 + j + 2);
        }
        ok = mbar_wait(&ctl, bar_full, ph, 55u);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        ph ^= 1u;
        tc_fence_after_sync();
        // index of the row's own position among this group's 128 columns: the columns up to it are seen by
        // a query row (statistics), the columns from it on see a key row (column sums)
        const int d = rt * kRows + row - (ct0 + j) * kCols - half * 128;
        const bool none = __all_sync(0xffffffffu, kSums ? d > 127 : d < 0);
        if (none) {
          tc_fence_before_sync();
          mbar_arrive(bar_empty);
          continue;
        }
        const bool full = __all_sync(0xffffffffu, kSums ? d <= 0 : d >= 127);
        uint32_t ra[32], rb[32];
        auto fold32 = [&](uint32_t (&r)[32], int c0) {
          if (!full) {
#pragma unroll
            for (int e = 0; e < 32; ++e)
              if (kSums ? c0 + e < d : c0 + e > d) r[e] = 0xff800000u;  // -inf
          }
          if (kSums) {
            const float* nl = nlse2_s[warp] + c0;
#pragma unroll
            for (int e = 0; e < 32; e += 4) {
              const ulonglong2 n4 = *reinterpret_cast<const ulonglong2*>(nl + e);
              const f32x2 x0 = fma2(pack2(r[e], r[e + 1]), sc, n4.x), x1 = fma2(pack2(r[e + 2], r[e + 3]), sc, n4.y);
              acc0 = add_exp2_pair<false>(acc0, x0, e / 2);
              acc1 = add_exp2_pair<false>(acc1, x1, e / 2 + 1);
            }
          } else {
            float m0 = -INFINITY, m1 = -INFINITY, m2 = -INFINITY, m3 = -INFINITY;
#pragma unroll
            for (int e = 0; e < 32; e += 4) {
              m0 = fmaxf(m0, __uint_as_float(r[e + 0]));
              m1 = fmaxf(m1, __uint_as_float(r[e + 1]));
              m2 = fmaxf(m2, __uint_as_float(r[e + 2]));
              m3 = fmaxf(m3, __uint_as_float(r[e + 3]));
            }
            const float m_new = fmaxf(ml.x, fmaxf(fmaxf(m0, m1), fmaxf(m2, m3)) * a.scale2);
            const f32x2 nr = pack2(-m_new);
            f32x2 s0 = 0ull, s1 = 0ull;
#pragma unroll
            for (int e = 0; e < 32; e += 4) {
              const f32x2 x0 = fma2(pack2(r[e], r[e + 1]), sc, nr), x1 = fma2(pack2(r[e + 2], r[e + 3]), sc, nr);
              s0 = add_exp2_pair<false>(s0, x0, e / 2);
              s1 = add_exp2_pair<false>(s1, x1, e / 2 + 1);
            }
            const float2 v = unpack2(add2(s0, s1));
            ml.y = fmaf(ml.y, ex2_approx(ml.x - m_new), v.x + v.y);
            ml.x = m_new;
          }
        };
        tmem_ld32_issue(taddr, ra);
#pragma unroll
        for (int c0 = 0; c0 < 128; c0 += 64) {
          tmem_ld_wait(ra);
          tmem_ld32_issue(taddr + c0 + 32, rb);
          fold32(ra, c0);
          tmem_ld_wait(rb);
          if (c0 == 0) {
            tmem_ld32_issue(taddr + 64, ra);
          } else {
            tc_fence_before_sync();
            mbar_arrive(bar_empty);  // the accumulator is in registers: hand the buffer back early
          }
          fold32(rb, c0 + 32);
        }
      }
      if (!ok) break;
      // the four groups' parts of a row meet in shared memory, double-buffered over the items
      const int xslot = n & 1;
      if (kSums) {
        const float2 v = unpack2(add2(acc0, acc1));
        nan_at = __reduce_max_sync(0xffffffffu, nan_at);
        ml = make_float2(0.f, nan_at >= rt * kRows + row ? __uint_as_float(0x7fc00000u) : v.x + v.y);
      }
      if (grp != 0) {
        ok = __all_sync(0xffffffffu, mbar_wait(&ctl, x_empty(xslot), ((n >> 1) & 1) ^ 1, 56u));
        if (!ok) break;
        xs[xslot][grp - 1][row] = ml;
        mbar_arrive(x_full(xslot));
      } else {
        ok = __all_sync(0xffffffffu, mbar_wait(&ctl, x_full(xslot), (n >> 1) & 1, 57u));
        if (!ok) break;
        float2 o[kGroups - 1];
        float m = ml.x;
#pragma unroll
        for (int g = 0; g < kGroups - 1; ++g) { o[g] = xs[xslot][g][row]; m = fmaxf(m, o[g].x); }
        mbar_arrive(x_empty(xslot));
        const int t = rt * kRows + row;
        float out;
        if (kSums) {
          out = (ml.y + o[0].y) + (o[1].y + o[2].y);
        } else {
          float l = ml.y * ex2_approx(ml.x - m);
#pragma unroll
          for (int g = 0; g < kGroups - 1; ++g) l = fmaf(o[g].y, ex2_approx(o[g].x - m), l);
          out = m + log2f(l);
        }
        if (t < a.L) (kSums ? a.part : a.lse2)[(size_t)head * a.L + t] = out;
      }
      j0 += n_jobs;
    }
    // a wait that ran out (a bug or a failing device) must not pass for a result: the rows that are missing become NaN
    if (!ok && grp == 0)
      for (; item_at<kSums>(a, n, head, rt, ct0, n_jobs); ++n)
        if (rt * kRows + row < a.L)
          (kSums ? a.part : a.lse2)[(size_t)head * a.L + rt * kRows + row] = __uint_as_float(0x7fc00000u);
  }

  // ---------------------------------------------------------------- teardown (every path)
  if (ctl.abort) {
    for (int i = 0; i < 50; ++i) __nanosleep(20000);  // let TMA copies still in flight land
  }
  tc_fence_before_sync();
  __syncthreads();
  pdl_trigger();
  if (warp == kMmaWarp) tmem_dealloc(tmem_base, 512);
}

// score[b, h, t]: the parts of the group's query heads, in their order
__global__ void __launch_bounds__(256)
accum_group_sum_kernel(const float* __restrict__ part, float* __restrict__ scores, int G, int L) {
  pdl_trigger();
  pdl_wait();
  const int t = blockIdx.x * 256 + threadIdx.x, unit = blockIdx.y;
  if (t >= L) return;
  float x = 0.f;
  for (int g = 0; g < G; ++g) x += part[((size_t)unit * G + g) * L + t];
  scores[(size_t)unit * L + t] = x;
}

template <bool kSums>
cudaError_t launch_pass(const AccumArgs& a, const CUtensorMap& am, const CUtensorMap& bm, cudaStream_t st) {
  static OncePerDevice granted;
  cudaError_t e = grant_smem(accum_tc_kernel<kSums>, kSmem, granted);
  if (e != cudaSuccess) return e;
  return launch_pdl(accum_tc_kernel<kSums>, dim3(a.items < kSms ? a.items : kSms), dim3(kThreads), (size_t)kSmem, st, am, bm, a);
}

size_t rows_bytes(int B, int Hq, int L) { return ((size_t)B * Hq * L * 4 + 255) / 256 * 256; }

}  // namespace

// Row statistics, the heads' parts, and a word where the bounded waits leave their code.  No entry point reads it and
// nothing clears it: a wait that ran out shows as NaN rows.
size_t accum_scores_workspace_bytes(int B, int Hq, int L) { return 2 * rows_bytes(B, Hq, L) + 256; }

cudaError_t launch_accum_scores(int B, int Hq, int Hkv, int L, float scale2, const void* Q_full, const void* K,
                                char* wsp, float* scores, cudaStream_t st) {
  AccumArgs a{};
  a.Hq = Hq; a.G = Hq / Hkv; a.L = L; a.heads = B * Hq;
  a.n_rt = (L + kRows - 1) / kRows;
  a.n_ct = (L + kCols - 1) / kCols;
  a.items = a.heads * a.n_rt;
  a.scale2 = scale2;
  a.lse2 = (float*)wsp;
  a.part = (float*)(wsp + rows_bytes(B, Hq, L));
  a.status = (unsigned*)(wsp + 2 * rows_bytes(B, Hq, L));
  CUtensorMap qa, qb, ka, kb;
  const uint64_t qd[2] = {(uint64_t)L, (uint64_t)a.heads}, kd[2] = {(uint64_t)L, (uint64_t)B * Hkv};
  const uint64_t str[2] = {256, (uint64_t)L * 256};
  const uint32_t abox[2] = {kRows, 1}, bbox[2] = {kCols, 1};
  if (!make_tensor_map_bf16(&qa, Q_full, 3, qd, str, abox) || !make_tensor_map_bf16(&qb, Q_full, 3, qd, str, bbox) ||
      !make_tensor_map_bf16(&ka, K, 3, kd, str, abox) || !make_tensor_map_bf16(&kb, K, 3, kd, str, bbox))
    return cudaErrorInvalidValue;
  cudaError_t e = launch_pass<false>(a, qa, kb, st);
  if (e == cudaSuccess) e = launch_pass<true>(a, ka, qb, st);
  if (e == cudaSuccess)
    e = launch_pdl(accum_group_sum_kernel, dim3((L + 255) / 256, B * Hkv), dim3(256), 0, st, (const float*)a.part, scores,
                   a.G, L);
  if (e != cudaSuccess) return e;
  count_launch(3);
  return cudaGetLastError();
}

}  // namespace calidrop
