"""GPU parity: the CUDA path through the C-ABI against the fp64 oracle, element by element.

Tolerances: kept-index sets bit-exact except near-tie swaps
(oracle pooled votes within 1e-5 relative); K_kept/V_kept/C_q bit-exact; O_c and decode
outputs within max-abs 2e-2 and mean-abs 2e-3; LSE_c and the output LSE within 1e-3.
"""
import os
import subprocess
import sys
import threading

import numpy as np
import pytest
import torch

import oracle
from paper_2507_19906_b200 import workload as wl

from gpu_util import (assert_close_lse, assert_close_out, check_kept_sets, compare_compress, decode_steps_compare,
                      gpu_compress, to_bits, to_dev)

pytestmark = pytest.mark.gpu


def _inputs(cfg, layer=0):
    Q = wl.gen_q_obs(cfg, layer)
    K, V = wl.gen_kv(cfg, layer)
    return Q, K, V


# ---------------------------------------------------------------- small shapes, every step
SMALL = [
    # B, Hq, Hkv, L, W, pool, budget, n_cal
    (1, 1, 1, 140, 1, 1, 9, 1),          # single window row, no pooling
    (1, 4, 2, 300, 8, 5, 40, 1),         # Algorithm 1 as printed (last query only)
    (2, 8, 2, 517, 16, 7, 100, 16),      # ragged L, G = 4, every window row calibrates
    (1, 7, 1, 1000, 32, 7, 128, 5),      # G = 7
    (1, 8, 1, 259, 4, 3, 30, 2),         # G = 8
    (2, 6, 3, 1301, 32, 5, 64, 32),      # spans several 128-key tiles with a ragged tail
    (1, 4, 4, 130, 64, 7, 65, 64),       # L - W < one tile, k_sel = 1
    (1, 2, 1, 96, 8, 7, 95, 3),          # a single evicted candidate
    (1, 7, 1, 700, 64, 7, 160, 64),      # 448 window rows per kv head: two row blocks in the vote pass
    (1, 16, 2, 900, 64, 5, 200, 16),     # G = 8, W = 64: 512 window rows, four 128-row statistic blocks
    (1, 4, 1, 3000, 128, 7, 400, 128),   # W = 128: one query head per calibration row block
    (1, 8, 1, 4000, 16, 7, 2100, 16),    # one unit: one cluster of eight CTAs, 263 rows each
    (2, 8, 2, 2500, 16, 7, 1000, 7),     # four units: most CTAs without a C_q row
    (1, 8, 1, 1500, 128, 7, 400, 4),     # 1024 window rows per kv head: the CUDA-core scoring and calibration kernels
    (1, 2, 1, 1200, 160, 5, 400, 160),   # window of 160 rows (beyond the 128-row tiles): the same kernels, n_cal = W
]


@pytest.mark.parametrize("B,Hq,Hkv,L,W,pool,budget,n_cal", SMALL)
def test_compress_and_decode_small(cuda_lib, B, Hq, Hkv, L, W, pool, budget, n_cal):
    cfg = wl.small_config(B=B, Hq=Hq, Hkv=Hkv, L=L, window=W, pool=pool, budget=budget, steps=5,
                          n_sink=2, n_heavy=max(1, L // 50))
    Q, K, V = _inputs(cfg)
    T = 5
    g = gpu_compress(Q, K, V, window=W, pool=pool, budget=budget, n_cal=n_cal, cap=budget + T)
    orc = oracle.compress(Q, K, V, window=W, pool=pool, budget=budget, n_cal=n_cal, cap=budget + T)
    # intermediate arrays, for a sharper diagnosis than the kept set alone
    np.testing.assert_allclose(g.row_lse, orc.row_lse, atol=2e-5)
    np.testing.assert_allclose(g.vote, orc.vote, rtol=2e-5, atol=1e-9)
    np.testing.assert_allclose(g.pooled, orc.pooled, rtol=2e-5, atol=1e-9)
    ref, _ = compare_compress(g, Q, K, V, window=W, pool=pool, budget=budget, n_cal=n_cal, orc=orc)
    q, kn, vn = wl.gen_decode_inputs(cfg, Q, steps=T)
    st = decode_steps_compare(g, ref, q, kn, vn, steps=T)
    assert st["total"] == T * B * Hq


def test_single_cta_selection_for_very_long_prompts(cuda_lib):
    """Beyond 262144 tokens the eight-CTA cluster selection no longer holds a unit's keys in registers
    and the single-CTA radix selection takes over; everything else is the usual path."""
    L, W, pool, budget, n_cal = 263000, 8, 7, 1000, 2
    cfg = wl.small_config(B=1, Hq=1, Hkv=1, L=L, window=W, pool=pool, budget=budget, steps=2, n_sink=4, n_heavy=300)
    Q, K, V = _inputs(cfg)
    g = gpu_compress(Q, K, V, window=W, pool=pool, budget=budget, n_cal=n_cal, cap=budget + 2)
    orc = oracle.compress(Q, K, V, window=W, pool=pool, budget=budget, n_cal=n_cal, cap=budget + 2)
    np.testing.assert_allclose(g.pooled, orc.pooled, rtol=2e-5, atol=1e-9)
    ref, _ = compare_compress(g, Q, K, V, window=W, pool=pool, budget=budget, n_cal=n_cal, orc=orc)
    q, kn, vn = wl.gen_decode_inputs(cfg, Q, steps=2)
    decode_steps_compare(g, ref, q, kn, vn, steps=2)


@pytest.mark.parametrize("units,G,W,L,own_kernel", [
    (3, 1, 8, 300, False),        # combined by the votes: 32 threads share a row, two statistics tiles
    (2, 8, 64, 700, False),       # ... 512 rows in two virtual units, a thread each
    (40, 4, 16, 1500, False),     # ... CTAs whose range spans two units
    (1, 4, 32, 20000, True),      # too many partials for it: a kernel of its own
    (300, 1, 8, 140, True),       # ... CTAs of more than two units
    (1, 4, 32, 20225, True),      # one unit: 80 tiles on a CTA each, 81 slots of four partials
    (1, 4, 64, 32768, True),      # ... 129 slots of two
    (1, 1, 8, 32768, True),       # ... of four
    (1, 2, 16, 65536, True),      # ... two tiles a CTA
])
def test_row_lse_of_the_statistics(cuda_lib, units, G, W, L, own_kernel):
    """Row LSE that a compress call leaves in its workspace, against fp64.  A logit is a sum of 128 exact products in
    fp32: an error of 128 * 2^-24 of a sum of magnitudes below 13 at the most, 1e-4.  (A pool wider than the cluster kernel's
    halo keeps the calls on the separate kernels.)"""
    cd = cuda_lib
    gen = torch.Generator(device="cuda").manual_seed(L)
    rn = lambda *sh: torch.randn(sh, generator=gen, device="cuda").to(torch.bfloat16)
    Q, K, V = rn(1, units * G, W, 128), rn(1, units, L, 128), rn(1, units, L, 128)
    p = cd.make_params(B=1, Hq=units * G, Hkv=units, L=L, window=W, pool=131, budget=W + 20, n_cal=1, cap=W + 20)
    st = cd.alloc_layer_state(p)
    before = cd.calidrop_launch_count()
    cd.calidrop_compress(p, Q, K, V, None, st.kept_idx, st.K_kept, st.V_kept, st.O_c, st.LSE_c, st.C_q, st.ws_compress)
    torch.cuda.synchronize()
    # statistics, (row LSE,) votes, selection, calibration, its reduction with the compaction
    assert cd.calidrop_launch_count() - before == (6 if own_kernel else 5)
    off = cd.calidrop_compress_workspace_layout(p).row_lse_offset
    got = st.ws_compress[off:off + units * G * W * 4].view(torch.float32).view(units, G * W)
    s = torch.einsum("urd,utd->urt", Q.view(units, G * W, 128).double(), K[0].double()) / 128 ** 0.5
    last = L - W + torch.arange(G * W, device="cuda") % W
    s.masked_fill_(torch.arange(L, device="cuda")[None, None] > last[None, :, None], -float("inf"))
    assert (got.double() - torch.logsumexp(s, -1)).abs().max() < 1e-4


@pytest.mark.parametrize("gap_one,gap_rest", [(78, 78), (78, 140), (140, 140)])
@pytest.mark.parametrize("G,W,one_kernel", [(2, 16, True), (4, 40, False)])
def test_calibration_of_evicted_rows_with_almost_no_attention(cuda_lib, gap_one, gap_rest, G, W, one_kernel):
    """The kept rows lead the evicted ones by `gap` nats, one row per kv head by another gap.  A probability below 2^-126
    is 0 and adds nothing; where all of them are, the row has no calibration: O_c = 0, LSE_c = -inf, not applied.  The
    one row at 78 nats is e^-82 of the softmax, far from the rest at e^-144."""
    cd = cuda_lib
    units, L, n_heavy = 2, 3000, 64
    gen = torch.Generator(device="cuda").manual_seed(gap_one + gap_rest)
    rn = lambda *sh: torch.randn(sh, generator=gen, device="cuda")
    e = rn(units, 128).sign()
    Q = (2.0 * e[None, :, None, None, :]).expand(1, units, G, W, 128).reshape(1, units * G, W, 128).to(torch.bfloat16)
    level = torch.full((units, L), -gap_rest / 2.0, device="cuda")
    level[:, L - W:] = 0.0
    at = torch.randperm(L - W, generator=gen, device="cuda")
    level[:, at[:n_heavy]] = gap_rest / 2.0
    level[:, at[n_heavy]] = gap_rest / 2.0 - gap_one
    # a key of `a` times the signs has the logit 2 a 128 / sqrt(128)
    K = ((level / (2 * 128 ** 0.5))[..., None] * e[:, None]).to(torch.bfloat16)[None].contiguous()
    V = rn(1, units, L, 128).to(torch.bfloat16)
    budget = W + n_heavy
    p = cd.make_params(B=1, Hq=units * G, Hkv=units, L=L, window=W, pool=1, budget=budget, n_cal=W, cap=budget, theta2=-1.0)
    st = cd.alloc_layer_state(p)
    before = cd.calidrop_launch_count()
    cd.calidrop_compress(p, Q, K, V, None, st.kept_idx, st.K_kept, st.V_kept, st.O_c, st.LSE_c, st.C_q, st.ws_compress)
    assert (cd.calidrop_launch_count() - before == 1) == one_kernel
    assert torch.equal(st.kept_idx[0, :, :n_heavy].long(), at[:n_heavy].sort().values.expand(units, -1))
    out = torch.empty((1, units * G, 128), dtype=torch.bfloat16, device="cuda")
    flags = torch.empty((1, units * G), dtype=torch.uint8, device="cuda")
    cd.calidrop_decode(p, Q[:, :, -1].contiguous(), None, None, st.K_kept, st.V_kept, budget, st.O_c, st.LSE_c, st.C_q, out,
                       None, flags, st.ws_decode)
    if gap_one > 100:
        assert torch.all(st.LSE_c == -float("inf")) and not st.O_c.any() and not (flags & 1).any()
        return
    evicted = torch.ones(L, dtype=torch.bool, device="cuda")
    evicted[L - W:] = False
    evicted[at[:n_heavy]] = False
    s = torch.einsum("urd,utd->urt", Q.view(units, G * W, 128).double(), K[0].double())[..., evicted] / 128 ** 0.5
    assert (st.LSE_c.view(units, G * W).double() - torch.logsumexp(s, -1)).abs().max() < 1e-3
    want = torch.softmax(s, -1) @ V[0][:, evicted].double()
    assert (st.O_c.view(units, G * W, 128).double() - want).abs().max() < 2e-2
    assert (flags & 1).all()


@pytest.mark.parametrize("G,W,one_kernel", [(4, 8, True), (4, 40, False)])
def test_votes_with_a_row_lse_far_below_the_logits(cuda_lib, G, W, one_kernel):
    """A caller's row LSE is not validated: one row's that is 200 nats too low makes every vote overflow to infinity,
    whichever of the 32 columns the row is, and the lowest candidates win."""
    cd = cuda_lib
    gen = torch.Generator(device="cuda").manual_seed(5)
    rn = lambda *sh: torch.randn(sh, generator=gen, device="cuda").to(torch.bfloat16)
    L, budget = 900, 60
    Q, K, V = rn(1, G, W, 128), rn(1, 1, L, 128), rn(1, 1, L, 128)
    p = cd.make_params(B=1, Hq=G, Hkv=1, L=L, window=W, pool=1, budget=budget, n_cal=1, cap=budget)
    st = cd.alloc_layer_state(p)
    off = cd.calidrop_compress_workspace_layout(p).vote_offset
    for row in range(G * W):
        lse = torch.full((G * W,), 7.0, device="cuda")
        lse[row] = -200.0
        before = cd.calidrop_launch_count()
        cd.calidrop_compress(p, Q, K, V, lse.view(1, G, W), st.kept_idx, st.K_kept, st.V_kept, st.O_c, st.LSE_c, st.C_q,
                             st.ws_compress)
        assert (cd.calidrop_launch_count() - before == 1) == one_kernel
        votes = st.ws_compress[off:off + 4 * (L - W)].view(torch.float32)
        assert torch.all(votes == float("inf")), row
        assert torch.equal(st.kept_idx[0, 0, :budget - W].long(), torch.arange(budget - W, device="cuda"))


@pytest.mark.parametrize("G,W,one_kernel", [(4, 8, True), (4, 40, False)])
def test_nan_inputs_leave_a_nan_wherever_they_lie(cuda_lib, G, W, one_kernel):
    """One NaN in a key or query row reaches every result that depends on it, at every position inside the 32 logits that
    a thread works on at a time: row LSE, votes, accumulated scores; a calibration over such a key is none."""
    cd = cuda_lib
    gen = torch.Generator(device="cuda").manual_seed(9)
    rn = lambda *sh: torch.randn(sh, generator=gen, device="cuda").to(torch.bfloat16)
    L, budget = 300, 60
    Q, K, V, Q_full = rn(1, G, W, 128), rn(1, 1, L, 128), rn(1, 1, L, 128), rn(1, G, L, 128)
    p = cd.make_params(B=1, Hq=G, Hkv=1, L=L, window=W, pool=1, budget=budget, n_cal=W, cap=budget)
    st = cd.alloc_layer_state(p)
    lay = cd.calidrop_compress_workspace_layout(p)
    get = lambda off, n: st.ws_compress[off:off + 4 * n].view(torch.float32)
    lse = torch.full((1, G, W), 7.0, device="cuda")
    outs = (st.K_kept, st.V_kept, st.O_c, st.LSE_c, st.C_q, st.ws_compress)
    scores = torch.empty((1, 1, L), device="cuda")
    ws = torch.empty((cd.calidrop_accumulated_scores_workspace_bytes(p),), dtype=torch.uint8, device="cuda")
    kept = torch.arange(L - budget, L, dtype=torch.int32, device="cuda").view(1, 1, budget)
    for t in range(32):
        Kt, Qt = K.clone(), Q.clone()
        Kt[0, 0, 32 + t, 5] = float("nan")
        Qt.view(G * W, 128)[t, 5] = float("nan")
        before = cd.calidrop_launch_count()
        cd.calidrop_compress(p, Q, Kt, V, None, st.kept_idx, *outs)
        assert (cd.calidrop_launch_count() - before == 1) == one_kernel
        assert torch.all(torch.isnan(get(lay.row_lse_offset, G * W))), t
        cd.calidrop_compress(p, Qt, K, V, lse, st.kept_idx, *outs)
        assert torch.all(torch.isnan(get(lay.vote_offset, L - W))), t
        cd.calidrop_calibrate(p, Q, Kt, V, lse, kept, *outs)
        assert torch.all(st.LSE_c == -float("inf")) and not st.O_c.any(), t
        cd.calidrop_accumulated_scores(p, Q_full, Kt, scores, ws)
        assert torch.all(torch.isnan(scores)), t


@pytest.mark.parametrize("L", [100, 300, 650])
def test_nan_query_reaches_the_keys_it_sees_only(cuda_lib, L):
    """Accumulated scores with a NaN in one query row: NaN up to its own position, as without it from there on."""
    cd = cuda_lib
    gen = torch.Generator(device="cuda").manual_seed(L)
    rn = lambda *sh: torch.randn(sh, generator=gen, device="cuda").to(torch.bfloat16)
    G = 2
    Q, K = rn(1, G, L, 128), rn(1, 1, L, 128)
    p = cd.make_params(B=1, Hq=G, Hkv=1, L=L, window=1, pool=1, budget=L, n_cal=1, cap=L)
    want, got = (torch.empty((1, 1, L), device="cuda") for _ in range(2))
    ws = torch.empty((cd.calidrop_accumulated_scores_workspace_bytes(p),), dtype=torch.uint8, device="cuda")
    cd.calidrop_accumulated_scores(p, Q, K, want, ws)
    for i in [0, 1, 10, 31, 32, 63, 64, 127, 128, 129, 255, 256, 300, 511, L - 1]:
        if i >= L:
            continue
        Qn = Q.clone()
        Qn[0, 1, i, 77] = float("nan")
        cd.calidrop_accumulated_scores(p, Qn, K, got, ws)
        assert torch.all(torch.isnan(got[0, 0, :i + 1])), i
        assert torch.equal(got[0, 0, i + 1:], want[0, 0, i + 1:]), i


@pytest.mark.parametrize("units,L,tail,pool,budget", [
    (1, 2048, 7, 1, 100),          # a full single CTA
    (3, 2049, 1, 7, 2048),         # the second CTA of the cluster holds one window row and no candidate
    (2, 16384, 16, 5, 600),        # eight CTAs of 512 x 4, full
    (2, 16385, 16, 3, 16384),      # five CTAs of 512 x 8, one row evicted
    (40, 16390, 8, 7, 64),         # more clusters than fit at 4 and 8 keys per thread
    (1, 70000, 32, 131, 5000),     # 1024 threads x 16 keys, a pool wider than the staged halo
    (1, 140000, 32, 9, 40000),     # 1024 threads x 32 keys
])
@pytest.mark.parametrize("ties", [False, True])
def test_selection_from_scores_at_the_edges_of_its_launch_shapes(cuda_lib, units, L, tail, pool, budget, ties):
    """Kept lists against a stable sort.  The scores are multiples of 2^-6 below 8 (`ties`: only eight distinct
    values, whole runs equal to the threshold), so every pooled sum is exact and the order has no rounding."""
    cd = cuda_lib
    rng = np.random.Generator(np.random.Philox(key=[61, L + ties]))
    scores = rng.integers(0, 8 if ties else 512, size=(1, units, L)).astype(np.float32) / 64
    p = cd.make_params(B=1, Hq=units, Hkv=units, L=L, window=min(tail, 8), pool=pool, budget=budget, n_cal=1, cap=budget)
    ws = torch.empty((cd.calidrop_compress_workspace_bytes(p),), dtype=torch.uint8, device="cuda")
    kept = torch.full((1, units, budget), -1, dtype=torch.int32, device="cuda")
    cd.calidrop_select_from_scores(p, torch.from_numpy(scores).cuda(), tail, kept, ws)
    got = kept.cpu().numpy()[0]
    n = L - tail
    for u in range(units):
        csum = np.concatenate([[0.0], np.cumsum(scores[0, u, :n].astype(np.float64))])
        t = np.arange(n)
        pooled = csum[np.minimum(t + pool // 2 + 1, n)] - csum[np.maximum(t - pool // 2, 0)]
        want = np.sort(np.argsort(-pooled, kind="stable")[:budget - tail])
        np.testing.assert_array_equal(got[u], np.concatenate([want, np.arange(n, L)]))


@pytest.mark.parametrize("units,L,tail,pool,budget", [
    (1, 32769, 1, 7, 300),         # five CTAs of 1024 x 8, the last with one window row only
    (2, 131072, 64, 5, 4096),      # sixteen CTAs, full
    (1, 131073, 9, 1, 131000),     # nine CTAs of 1024 x 16
    (40, 33000, 8, 7, 64),         # more clusters of sixteen than run at once: eight CTAs of 512 x 16
    (30, 66000, 8, 3, 500),        # ... of 1024 x 16
])
def test_selection_on_clusters_of_more_than_eight(cuda_lib, units, L, tail, pool, budget):
    """As above, with the clusters of up to sixteen CTAs that long prompts of few units get, and past their edge."""
    test_selection_from_scores_at_the_edges_of_its_launch_shapes(cuda_lib, units, L, tail, pool, budget, False)


@pytest.mark.parametrize("calib_size", [1, 40, 300, 10 ** 6, -1])
@pytest.mark.parametrize("B,Hq,Hkv,L,W,budget,n_cal,one_kernel", [
    (2, 8, 2, 1500, 16, 200, 16, True),
    (1, 8, 2, 1500, 64, 200, 16, False),      # 256 window rows: the separate kernels
    (1, 150, 150, 400, 16, 200, 4, False),    # more units than the device holds clusters
])
def test_calibration_size(cuda_lib, calib_size, B, Hq, Hkv, L, W, budget, n_cal, one_kernel):
    """Section 4.4's calibration size m: only the m evicted rows of highest pooled vote are calibrated
    (and offloaded); m >= the number evicted is Algorithm 1 as printed, -1 switches the calibration off."""
    from paper_2507_19906_b200 import binding as cd
    pool = 7
    cfg = wl.small_config(B=B, Hq=Hq, Hkv=Hkv, L=L, window=W, pool=pool, budget=budget, steps=3, n_sink=2, n_heavy=40)
    Q, K, V = _inputs(cfg)
    m = None if calib_size == 10 ** 6 else max(calib_size, 0)
    orc = oracle.compress(Q, K, V, window=W, pool=pool, budget=budget, n_cal=n_cal, cap=budget + 3, calib_size=m)
    p = cd.make_params(B=B, Hq=Hq, Hkv=Hkv, L=L, window=W, pool=pool, budget=budget, n_cal=n_cal, cap=budget + 3,
                       calib_size=calib_size)
    st = cd.alloc_layer_state(p)
    dQ, dK, dV = to_dev(Q), to_dev(K), to_dev(V)
    before = cd.calidrop_launch_count()
    cd.calidrop_compress(p, dQ, dK, dV, None, st.kept_idx, st.K_kept, st.V_kept, st.O_c, st.LSE_c, st.C_q,
                         st.ws_compress)
    torch.cuda.synchronize()
    assert (cd.calidrop_launch_count() - before == 1) == (one_kernel and calib_size != -1)
    np.testing.assert_array_equal(st.kept_idx.cpu().numpy(), orc.kept_idx)      # no near-tie in this input
    np.testing.assert_array_equal(to_bits(st.C_q), orc.C_q)
    assert_close_lse(st.LSE_c.cpu().numpy(), orc.LSE_c, "LSE_c")
    assert_close_out(st.O_c.cpu().numpy(), orc.O_c, "O_c")
    if calib_size == -1:
        assert np.all(np.isneginf(st.LSE_c.cpu().numpy()))
        return
    # the calibrated rows, compacted for offloading: the same list and bit copies of the rows
    n_e = min(calib_size, L - budget)
    ev_idx = torch.empty((B, Hkv, n_e), dtype=torch.int32, device="cuda")
    K_e = torch.empty((B, Hkv, n_e, 128), dtype=torch.bfloat16, device="cuda")
    V_e = torch.empty_like(K_e)
    cd.calidrop_gather_evicted(p, dK, dV, st.kept_idx, ev_idx, K_e, V_e, st.ws_compress)
    torch.cuda.synchronize()
    want = orc.calib_idx if m is not None else np.stack(
        [[np.setdiff1d(np.arange(L - W), orc.kept_idx[b, h]) for h in range(Hkv)] for b in range(B)])
    np.testing.assert_array_equal(ev_idx.cpu().numpy(), want)
    for b in range(B):
        for h in range(Hkv):
            np.testing.assert_array_equal(to_bits(K_e)[b, h], K[b, h][want[b, h]])
            np.testing.assert_array_equal(to_bits(V_e)[b, h], V[b, h][want[b, h]])
    # and decode goes on as usual with the smaller calibration term
    g = type("R", (), {})()
    g.p, g.st, g.n_kept = p, st, budget
    ref = orc
    q, kn, vn = wl.gen_decode_inputs(cfg, Q, steps=3)
    decode_steps_compare(g, ref, q, kn, vn, steps=3)


ONE_KERNEL = [
    # B, Hq, Hkv, L, W, pool, budget, n_cal, calib_size, whether the cluster kernel takes it
    (1, 1, 1, 136, 8, 7, 40, 1, 0, True),           # two CTAs, the second has window rows only
    (1, 2, 1, 128 * 3 + 33, 32, 1, 70, 32, 0, True),   # 64 window rows (two copies of them on the lanes), one candidate in the last tile
    (1, 5, 1, 2048, 8, 9, 200, 8, 0, True),         # sixteen CTAs of a tile, 40 rows, a pool without a kernel of its own
    (2, 5, 1, 2300, 24, 129, 300, 24, 500, True),   # 120 rows, the widest pool that the kernel takes, a calibration size
    (1, 4, 1, 900, 32, 5, 899, 32, 0, True),        # a single evicted candidate, 128 calibration rows
    (3, 8, 8, 1300, 16, 7, 17, 1, 3, True),         # 24 units, 16 rows; one candidate kept, three calibrated
    (1, 100, 100, 300, 8, 7, 50, 8, 0, True),       # one CTA to a unit
    (1, 100, 100, 128 * 17 + 5, 8, 5, 60, 2, 40, True),   # ... of 18 tiles: the groups take tiles of their own in the votes
    (1, 3, 1, 900, 64, 7, 200, 3, 0, False),         # 192 rows: the separate kernels, the row LSE combined by the votes
    (1, 100, 100, 900, 128, 131, 300, 2, 0, False),  # a pool wider than the halo
]


@pytest.mark.parametrize("B,Hq,Hkv,L,W,pool,budget,n_cal,calib_size,one_kernel", ONE_KERNEL)
@pytest.mark.parametrize("octaves", [None, 0, 24, -40])
def test_compress_in_one_kernel(cuda_lib, B, Hq, Hkv, L, W, pool, budget, n_cal, calib_size, one_kernel, octaves):
    """Units that a cluster holds take one kernel.  With `octaves` the caller supplies the row LSE, less that many factors of
    two: the votes then lie inside, above and below the range that the first selection pass resolves.  Rounding the
    shifted row LSE moves a vote by 2^-18 of itself at most (|lse| below 64), the same for all keys of a row."""
    from paper_2507_19906_b200 import binding as cd
    cfg = wl.small_config(B=B, Hq=Hq, Hkv=Hkv, L=L, window=W, pool=pool, budget=budget, steps=1, n_sink=2,
                          n_heavy=max(1, L // 50))
    Q, K, V = _inputs(cfg)
    m = None if calib_size == 0 else calib_size
    orc = oracle.compress(Q, K, V, window=W, pool=pool, budget=budget, n_cal=n_cal, cap=budget, calib_size=m)
    p = cd.make_params(B=B, Hq=Hq, Hkv=Hkv, L=L, window=W, pool=pool, budget=budget, n_cal=n_cal, cap=budget,
                       calib_size=calib_size)
    st = cd.alloc_layer_state(p)
    dQ, dK, dV = to_dev(Q), to_dev(K), to_dev(V)
    lse = None
    if octaves is not None:
        lse = torch.from_numpy((orc.row_lse - octaves * np.log(2.0)).astype(np.float32)).cuda()
    before = cd.calidrop_launch_count()
    cd.calidrop_compress(p, dQ, dK, dV, lse, st.kept_idx, st.K_kept, st.V_kept, st.O_c, st.LSE_c, st.C_q, st.ws_compress)
    torch.cuda.synchronize()
    assert (cd.calidrop_launch_count() - before == 1) == one_kernel
    lay = cd.calidrop_compress_workspace_layout(p)
    assert int(st.ws_compress[lay.status_offset:lay.status_offset + 4].view(torch.int32).item()) == 0
    ws = lambda off, ref: st.ws_compress[off:off + 4 * ref.size].view(torch.float32).cpu().numpy().reshape(ref.shape)
    scale, rtol = 2.0 ** (octaves or 0), 2e-5 if not octaves else 4e-5
    np.testing.assert_allclose(ws(lay.vote_offset, orc.vote), orc.vote * scale, rtol=rtol, atol=1e-9 * scale)
    np.testing.assert_allclose(ws(lay.pooled_offset, orc.pooled), orc.pooled * scale, rtol=rtol, atol=1e-9 * scale)
    if octaves is None:
        np.testing.assert_allclose(ws(lay.row_lse_offset, orc.row_lse), orc.row_lse, atol=2e-5)
    kept = st.kept_idx.cpu().numpy()
    check_kept_sets(kept, orc)
    np.testing.assert_array_equal(to_bits(st.C_q), orc.C_q)
    for b in range(B):
        for h in range(Hkv):
            np.testing.assert_array_equal(to_bits(st.K_kept)[b, h], K[b, h][kept[b, h]])
            np.testing.assert_array_equal(to_bits(st.V_kept)[b, h], V[b, h][kept[b, h]])
    # the selection is that of the kernel's own pooled votes to the last bit, and the calibration state is that of the rows
    # it leaves (the shift of the row LSE does not enter)
    check_selection_and_calibration(p, st, dQ, dK, dV, ws(lay.pooled_offset, orc.pooled))


def check_selection_and_calibration(p, st, dQ, dK, dV, pooled):
    """Kept list and calibrated rows of a call against a stable sort of the pooled votes it left in its workspace, the calibration
    state against fp64 over those rows."""
    from paper_2507_19906_b200 import binding as cd
    B, Hkv, G, L, W, n_cal = p.B, p.Hkv, p.Hq // p.Hkv, p.L, p.window, p.n_cal
    k_sel, n_cand = p.budget - W, L - W
    m = n_cand - k_sel if p.calib_size == 0 else min(p.calib_size, n_cand - k_sel)
    order = np.argsort(-pooled.reshape(B * Hkv, n_cand), axis=-1, kind="stable")
    kept, calib = np.sort(order[:, :k_sel], -1), np.sort(order[:, k_sel:k_sel + m], -1)
    got = st.kept_idx.cpu().numpy().reshape(B * Hkv, p.budget)
    np.testing.assert_array_equal(got[:, :k_sel], kept)
    np.testing.assert_array_equal(got[:, k_sel:], np.broadcast_to(np.arange(n_cand, L), (B * Hkv, W)))
    ev_idx = torch.empty((B, Hkv, m), dtype=torch.int32, device="cuda")
    K_e, V_e = (torch.empty((B, Hkv, m, 128), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    cd.calidrop_gather_evicted(p, dK, dV, st.kept_idx, ev_idx, K_e, V_e, st.ws_compress)
    np.testing.assert_array_equal(ev_idx.cpu().numpy().reshape(B * Hkv, m), calib)
    q = dQ[:, :, W - n_cal:].reshape(B * Hkv, G * n_cal, 128).double()
    for u in range(B * Hkv):
        s = q[u] @ K_e.view(-1, m, 128)[u].double().T / 128 ** 0.5
        want_lse, want = torch.logsumexp(s, -1), torch.softmax(s, -1) @ V_e.view(-1, m, 128)[u].double()
        assert_close_lse(st.LSE_c.view(B * Hkv, -1)[u].cpu().numpy(), want_lse.cpu().numpy(), "LSE_c")
        assert_close_out(st.O_c.view(B * Hkv, -1, 128)[u].cpu().numpy(), want.cpu().numpy(), "O_c")


@pytest.mark.parametrize("units,L,W,G,pool", [
    (1, 2056, 8, 4, 1),         # CTAs of one or two tiles
    (3, 6000, 16, 8, 1),        # 128 window rows
    (100, 128 * 18 + 9, 8, 2, 1),   # one CTA of more than sixteen tiles to a unit
    (60, 128 * 40 - 3, 8, 2, 1),    # ... two
    (5, 3000, 8, 4, 3),         # pooled: runs of equal sums
])
@pytest.mark.parametrize("mid,low", [(0.5, 0.25), (0.5, -10.0)])
@pytest.mark.parametrize("sized", [False, True])
def test_ties_in_one_kernel(cuda_lib, units, L, W, G, pool, mid, low, sized):
    """Keys of three kinds, equal to the bit and so in their votes: the cut of the kept list lies inside the second kind, in the
    middle of the prompt, that of a calibration size inside the third, whose votes are in the range of the first selection pass
    or far below it."""
    cd = cuda_lib
    gen = torch.Generator(device="cuda").manual_seed(L + sized)
    rn = lambda *sh: torch.randn(sh, generator=gen, device="cuda")
    n_cand = L - W
    u = rn(units, 128).sign()
    Q = (u[:, None, None] * 0.5 + 0.1 * rn(units, G, W, 128)).reshape(1, units * G, W, 128).to(torch.bfloat16)
    kind = torch.rand((units, n_cand), generator=gen, device="cuda")
    kind = (kind > 0.1).long() + (kind > 0.4).long()                  # a tenth, three tenths, the rest
    level = torch.tensor([0.8, mid, low], device="cuda") / 2
    K = torch.cat([(level[kind][..., None] * u[:, None]), 0.1 * rn(units, W, 128)], 1).to(torch.bfloat16)[None].contiguous()
    V = rn(1, units, L, 128).to(torch.bfloat16)
    budget = W + n_cand // 4
    m = n_cand // 2 if sized else 0
    p = cd.make_params(B=1, Hq=units * G, Hkv=units, L=L, window=W, pool=pool, budget=budget, n_cal=2, cap=budget, calib_size=m)
    st = cd.alloc_layer_state(p)
    before = cd.calidrop_launch_count()
    cd.calidrop_compress(p, Q, K, V, None, st.kept_idx, st.K_kept, st.V_kept, st.O_c, st.LSE_c, st.C_q, st.ws_compress)
    torch.cuda.synchronize()
    assert cd.calidrop_launch_count() - before <= 2   # (the second one compacts many rows)
    off = cd.calidrop_compress_workspace_layout(p).pooled_offset
    pooled = st.ws_compress[off:off + 4 * units * n_cand].view(torch.float32).cpu().numpy().reshape(units, n_cand)
    if pool == 1:
        for row in pooled:
            assert len(np.unique(row)) == 3
    check_selection_and_calibration(p, st, Q, K, V, pooled)


@pytest.mark.parametrize("units,G,W,L,supply_lse,one_kernel", [
    (8, 4, 32, 8192, False, True),
    (8, 4, 32, 8192, True, True),
    (80, 4, 32, 3109, True, False),    # one CTA a unit: half of the SMs would be idle
    (80, 4, 32, 3109, False, True),
    (48, 5, 16, 8838, True, False),    # two CTAs a unit
])
def test_route_of_a_compress_call(cuda_lib, units, G, W, L, supply_lse, one_kernel):
    """The cluster kernel is taken where it was measured to be faster than the separate kernels."""
    cd = cuda_lib
    gen = torch.Generator(device="cuda").manual_seed(L)
    rn = lambda *sh: torch.randn(sh, generator=gen, device="cuda").to(torch.bfloat16)
    Q, K, V = rn(1, units * G, W, 128), rn(1, units, L, 128), rn(1, units, L, 128)
    lse = torch.full((1, units * G, W), 9.0, device="cuda") if supply_lse else None
    p = cd.make_params(B=1, Hq=units * G, Hkv=units, L=L, window=W, pool=7, budget=200, n_cal=1, cap=200)
    st = cd.alloc_layer_state(p)
    before = cd.calidrop_launch_count()
    cd.calidrop_compress(p, Q, K, V, lse, st.kept_idx, st.K_kept, st.V_kept, st.O_c, st.LSE_c, st.C_q, st.ws_compress)
    torch.cuda.synchronize()
    assert (cd.calidrop_launch_count() - before == 1) == one_kernel


@pytest.mark.parametrize("B,Hq,Hkv,L,W,pool,budget,n_cal", [c[:8] for c in ONE_KERNEL if c[8] == 0 and c[9]])
@pytest.mark.parametrize("supply_lse", [False, True])
def test_calibrate_in_one_kernel(cuda_lib, B, Hq, Hkv, L, W, pool, budget, n_cal, supply_lse):
    """The calibration for a given kept list takes the same cluster kernel without its selection: for the list that the whole
    step chose, the same rows and the same calibration state (the same sums in the same order)."""
    from paper_2507_19906_b200 import binding as cd
    cfg = wl.small_config(B=B, Hq=Hq, Hkv=Hkv, L=L, window=W, pool=pool, budget=budget, steps=1, n_sink=2,
                          n_heavy=max(1, L // 50))
    Q, K, V = (to_dev(x) for x in _inputs(cfg))
    p = cd.make_params(B=B, Hq=Hq, Hkv=Hkv, L=L, window=W, pool=pool, budget=budget, n_cal=n_cal, cap=budget)
    st, got = cd.alloc_layer_state(p), cd.alloc_layer_state(p)
    cd.calidrop_compress(p, Q, K, V, None, st.kept_idx, st.K_kept, st.V_kept, st.O_c, st.LSE_c, st.C_q, st.ws_compress)
    off = cd.calidrop_compress_workspace_layout(p).row_lse_offset
    lse = st.ws_compress[off:off + 4 * B * Hq * W].view(torch.float32).clone() if supply_lse else None
    before = cd.calidrop_launch_count()
    cd.calidrop_calibrate(p, Q, K, V, lse, st.kept_idx, got.K_kept, got.V_kept, got.O_c, got.LSE_c, got.C_q, got.ws_compress)
    torch.cuda.synchronize()
    assert cd.calidrop_launch_count() - before == 1
    lay = cd.calidrop_compress_workspace_layout(p)
    assert int(got.ws_compress[lay.status_offset:lay.status_offset + 4].view(torch.int32).item()) == 0
    for name in ("K_kept", "V_kept", "C_q"):
        assert torch.equal(getattr(got, name), getattr(st, name)), name
    assert torch.allclose(got.LSE_c, st.LSE_c, rtol=0, atol=1e-5) and torch.allclose(got.O_c, st.O_c, rtol=1e-5, atol=1e-6)


@pytest.mark.parametrize("units,L,W,budget,launches", [
    (100, 900, 8, 512, 1),      # one CTA to a unit: as many rows as the cluster kernel compacts itself
    (100, 900, 8, 513, 2),      # ... one more
    (60, 1500, 16, 1484, 2),    # two CTAs, sixteen evicted rows
    (60, 1500, 16, 1024, 1),
])
def test_compaction_of_many_rows_behind_the_cluster_kernel(cuda_lib, units, L, W, budget, launches):
    """Beyond 512 retained rows a CTA, a kernel of their own compacts them, for a chosen and for a given kept list."""
    from paper_2507_19906_b200 import binding as cd
    cfg = wl.small_config(B=1, Hq=units, Hkv=units, L=L, window=W, pool=5, budget=budget, steps=1, n_sink=2, n_heavy=20)
    Q, K, V = _inputs(cfg)
    before = cd.calidrop_launch_count()
    g = gpu_compress(Q, K, V, window=W, pool=5, budget=budget, n_cal=2, cap=budget + 3, keep_inputs=True)
    assert cd.calidrop_launch_count() - before == launches
    compare_compress(g, Q, K, V, window=W, pool=5, budget=budget, n_cal=2)
    got = cd.alloc_layer_state(g.p)
    before = cd.calidrop_launch_count()
    cd.calidrop_calibrate(g.p, to_dev(Q), g.dK, g.dV, None, g.st.kept_idx, got.K_kept, got.V_kept, got.O_c, got.LSE_c, got.C_q,
                          got.ws_compress)
    torch.cuda.synchronize()
    assert cd.calidrop_launch_count() - before == launches
    assert torch.equal(got.K_kept[:, :, :budget], g.st.K_kept[:, :, :budget])
    assert torch.equal(got.V_kept[:, :, :budget], g.st.V_kept[:, :, :budget])
    assert torch.allclose(got.LSE_c, g.st.LSE_c, rtol=0, atol=1e-5) and torch.allclose(got.O_c, g.st.O_c, rtol=1e-5, atol=1e-6)


@pytest.mark.parametrize("G,n_cal,octave", [(1, 1, 0), (2, 16, 0), (3, 16, 0), (4, 16, 0), (8, 16, 0), (2, 16, 200)])
def test_infinite_value_of_an_evicted_row_stays_infinite(cuda_lib, G, n_cal, octave):
    """The calibration rows of a small unit lie on the lanes two or four times, each copy with a part of the keys: an infinite
    value of V makes its column of O_c infinite (NaN where the probability is zero) and leaves every other element as it was."""
    from paper_2507_19906_b200 import binding as cd
    L, W, budget = 700, 16, 100
    cfg = wl.small_config(B=1, Hq=G, Hkv=1, L=L, window=W, pool=5, budget=budget, steps=1, n_sink=2, n_heavy=14)
    Q, K, V = (to_dev(x) for x in _inputs(cfg))
    p = cd.make_params(B=1, Hq=G, Hkv=1, L=L, window=W, pool=5, budget=budget, n_cal=n_cal, cap=budget)
    lse = None

    def run(V):
        st = cd.alloc_layer_state(p)
        before = cd.calidrop_launch_count()
        cd.calidrop_compress(p, Q, K, V, lse, st.kept_idx, st.K_kept, st.V_kept, st.O_c, st.LSE_c, st.C_q, st.ws_compress)
        torch.cuda.synchronize()
        assert cd.calidrop_launch_count() - before == 1
        off = cd.calidrop_compress_workspace_layout(p).row_lse_offset
        return st, st.ws_compress[off:off + 4 * G * W].view(torch.float32).clone()

    st, row_lse = run(V)
    if octave:   # the first row's probabilities are all zero
        lse = row_lse.clone()
        lse[W - 1] += octave
        lse = lse.view(1, G, W)
        st, _ = run(V)
    kept = set(st.kept_idx.flatten().tolist())
    evicted = [t for t in range(L - W) if t not in kept]
    for t in (evicted[0], evicted[len(evicted) // 2], evicted[-1]):
        Vi = V.clone()
        Vi[0, 0, t, 77] = -float("inf")
        got, _ = run(Vi)
        assert torch.equal(got.kept_idx, st.kept_idx) and torch.equal(got.LSE_c, st.LSE_c)
        col = got.O_c[0, :, :, 77].flatten()
        zero = torch.zeros_like(col, dtype=torch.bool)
        if octave:
            zero[n_cal - 1] = True
        assert torch.all(torch.isneginf(col[~zero])), t
        other = torch.arange(128, device="cuda") != 77
        assert torch.equal(got.O_c[..., other], st.O_c[..., other]), t


def test_infinite_values_of_all_evicted_rows(cuda_lib):
    """As above with an infinite value in every evicted row: of one sign the column of O_c is infinite, of both it is NaN, the
    other columns are as they were.  Settling the elements takes a bounded time (with a product of 128 terms per thread and
    key it took 11 ms where a call of finite values takes 0.04; now 0.8)."""
    cd = cuda_lib
    units, G, W, L, budget = 8, 8, 8, 8192, 108
    gen = torch.Generator(device="cuda").manual_seed(3)
    rn = lambda *sh: torch.randn(sh, generator=gen, device="cuda").to(torch.bfloat16)
    Q, K, V = rn(1, units * G, W, 128), rn(1, units, L, 128), rn(1, units, L, 128)
    p = cd.make_params(B=1, Hq=units * G, Hkv=units, L=L, window=W, pool=5, budget=budget, n_cal=W, cap=budget)

    def run(V):
        st = cd.alloc_layer_state(p)
        e = [torch.cuda.Event(enable_timing=True) for _ in range(4)]
        before = cd.calidrop_launch_count()
        for i in range(4):
            e[i].record()
            if i < 3:
                cd.calidrop_compress(p, Q, K, V, None, st.kept_idx, st.K_kept, st.V_kept, st.O_c, st.LSE_c, st.C_q, st.ws_compress)
        torch.cuda.synchronize()
        assert cd.calidrop_launch_count() - before == 3
        off = cd.calidrop_compress_workspace_layout(p).status_offset
        assert int(st.ws_compress[off:off + 4].view(torch.int32).item()) == 0
        return st, min(e[i].elapsed_time(e[i + 1]) for i in range(3))

    st, _ = run(V)
    evicted = torch.ones((units, L), dtype=torch.bool, device="cuda")
    evicted[:, L - W:] = False
    evicted.scatter_(1, st.kept_idx[0].long(), False)
    other = torch.arange(128, device="cuda") != 77
    for alternate in (False, True):
        Vi = V.clone()
        Vi[0, :, :, 77][evicted] = float("inf")
        if alternate:
            Vi[0, :, 1::2, 77] *= -1
        got, ms = run(Vi)
        assert torch.equal(got.kept_idx, st.kept_idx) and torch.equal(got.LSE_c, st.LSE_c)
        assert torch.all(torch.isnan(got.O_c[..., 77]) if alternate else torch.isposinf(got.O_c[..., 77]))
        assert torch.equal(got.O_c[..., other], st.O_c[..., other])
        assert ms < 4.0, ms


@pytest.mark.parametrize("Hkv,G,n", [(1, 2, 1997), (2, 8, 529), (8, 4, 1000), (1, 1, 33)])
def test_decode_with_an_infinite_value_in_any_row(cuda_lib, Hkv, G, n):
    """An infinite value of V in one row makes its column of the output infinite and touches no other, at whatever distance
    from the ends of the slices that a unit is cut into: no CTA may multiply a neighbour's rows by zero."""
    from paper_2507_19906_b200 import binding as cd
    g = torch.Generator(device="cuda").manual_seed(n)
    rn = lambda *sh: torch.randn(sh, generator=g, device="cuda")
    p = cd.make_params(B=1, Hq=G * Hkv, Hkv=Hkv, L=n + 64, window=16, pool=7, budget=n, n_cal=4, cap=n, theta2=-1.0)
    st = cd.alloc_layer_state(p)
    for t in (st.K_kept, st.V_kept, st.C_q, st.O_c, st.LSE_c):
        t.copy_(rn(*t.shape))
    q = rn(1, G * Hkv, 128).to(torch.bfloat16)
    lse, flags = torch.zeros((1, G * Hkv), device="cuda"), torch.zeros((1, G * Hkv), dtype=torch.uint8, device="cuda")

    def run():
        out = torch.zeros((1, G * Hkv, 128), dtype=torch.bfloat16, device="cuda")
        cd.calidrop_decode(p, q, None, None, st.K_kept, st.V_kept, n, st.O_c, st.LSE_c, st.C_q, out, lse, flags, st.ws_decode)
        return out

    clean = run()
    other = torch.arange(128, device="cuda") != 77
    ok = torch.ones((), dtype=torch.bool, device="cuda")
    for t in range(n):
        was = st.V_kept[0, :, t, 77].clone()
        st.V_kept[0, :, t, 77] = float("inf")
        out = run()
        ok &= torch.all(torch.isposinf(out[..., 77])) & torch.all(out[..., other] == clean[..., other])
        st.V_kept[0, :, t, 77] = was
    assert bool(ok)


def test_supplied_row_lse_matches_self_computed(cuda_lib):
    cfg = wl.small_config(B=1, Hq=4, Hkv=2, L=400, window=16, pool=7, budget=64)
    Q, K, V = _inputs(cfg)
    orc = oracle.compress(Q, K, V, window=16, pool=7, budget=64, n_cal=4)
    g = gpu_compress(Q, K, V, window=16, pool=7, budget=64, n_cal=4, lse_obs=orc.row_lse)
    compare_compress(g, Q, K, V, window=16, pool=7, budget=64, n_cal=4, orc=orc)


def test_budget_at_least_prefix_is_full_attention(cuda_lib):
    """Nothing evicted: LSE_c = -inf, O_c = 0, decode equals brute-force attention."""
    cfg = wl.small_config(B=1, Hq=4, Hkv=2, L=200, window=8, pool=5, budget=256)
    Q, K, V = _inputs(cfg)
    g = gpu_compress(Q, K, V, window=8, pool=5, budget=256, n_cal=2, cap=204)
    assert g.n_kept == 200
    np.testing.assert_array_equal(g.kept_idx, np.broadcast_to(np.arange(200), (1, 2, 200)))
    assert np.all(np.isneginf(g.LSE_c)) and np.all(g.O_c == 0)
    ref = oracle.compress(Q, K, V, window=8, pool=5, budget=256, n_cal=2, cap=204)
    q, kn, vn = wl.gen_decode_inputs(cfg, Q, steps=3)
    st = decode_steps_compare(g, ref, q, kn, vn, theta2=-1.0)
    assert st["applied"] == 0
    # and the GPU output against brute-force attention over the whole prompt plus the appended rows
    from paper_2507_19906_b200 import binding as cd
    out = torch.empty((1, 4, 128), dtype=torch.bfloat16, device="cuda")
    lse = torch.empty((1, 4), dtype=torch.float32, device="cuda")
    flags = torch.empty((1, 4), dtype=torch.uint8, device="cuda")
    # (the three steps above appended their rows to the GPU cache; repeat the last query without appending)
    cd.calidrop_decode(g.p, to_dev(q[2]), None, None, g.st.K_kept, g.st.V_kept, 203, g.st.O_c, g.st.LSE_c,
                       g.st.C_q, out, lse, flags, g.st.ws_decode)
    torch.cuda.synchronize()
    got = wl.bf16_bits_to_f64(to_bits(out))
    for hq in range(4):
        h = hq // 2
        Kf = np.concatenate([K[0, h], kn[:3, 0, h]])
        Vf = np.concatenate([V[0, h], vn[:3, 0, h]])
        o, l = oracle.full_attention(q[2, 0, hq][None], Kf, Vf)
        assert_close_out(got[0, hq], o[0], "nothing evicted: output vs brute-force full attention")
        assert abs(float(lse[0, hq]) - l[0]) < 1e-3


def test_query_equal_to_calibration_query_recovers_full_attention(cuda_lib):
    """Eq. 1's exact case on the GPU: q == C_q[c] => output == attention over the whole prompt."""
    cfg = wl.small_config(B=1, Hq=4, Hkv=2, L=600, window=16, pool=7, budget=80)
    Q, K, V = _inputs(cfg)
    n_cal = 4
    g = gpu_compress(Q, K, V, window=16, pool=7, budget=80, n_cal=n_cal)
    from paper_2507_19906_b200 import binding as cd
    out = torch.empty((1, 4, 128), dtype=torch.bfloat16, device="cuda")
    lse = torch.empty((1, 4), dtype=torch.float32, device="cuda")
    flags = torch.empty((1, 4), dtype=torch.uint8, device="cuda")
    for c in range(n_cal):
        qc = np.ascontiguousarray(Q[:, :, 16 - n_cal + c])
        cd.calidrop_decode(g.p, to_dev(qc), None, None, g.st.K_kept, g.st.V_kept, 80, g.st.O_c, g.st.LSE_c,
                           g.st.C_q, out, lse, flags, g.st.ws_decode)
        torch.cuda.synchronize()
        got = wl.bf16_bits_to_f64(to_bits(out))
        f = flags.cpu().numpy()
        assert np.all(f & 1 == 1) and np.all(f >> 2 == c)
        for hq in range(4):
            o, l = oracle.full_attention(qc[0, hq][None], K[0, hq // 2], V[0, hq // 2])
            assert_close_out(got[0, hq], o[0], "merged output vs brute-force full attention")
            assert abs(float(lse[0, hq]) - l[0]) < 1e-3


def test_gate_thresholds(cuda_lib):
    cfg = wl.small_config(B=2, Hq=4, Hkv=2, L=300, window=8, pool=5, budget=40)
    Q, K, V = _inputs(cfg)
    g = gpu_compress(Q, K, V, window=8, pool=5, budget=40, n_cal=8, cap=48)
    ref, _ = compare_compress(g, Q, K, V, window=8, pool=5, budget=40, n_cal=8)
    q, kn, vn = wl.gen_decode_inputs(cfg, Q, steps=2)
    never = decode_steps_compare(g, ref, q, kn, vn, theta1=0.0, theta2=1.0, steps=1, append=False)
    always = decode_steps_compare(g, ref, q, kn, vn, theta1=0.0, theta2=-1.0, steps=1, append=False)
    assert never["applied"] == 0 and always["applied"] == always["total"]
    paper = decode_steps_compare(g, ref, q, kn, vn, theta1=0.7, theta2=0.85, steps=2, append=True)
    assert paper["total"] == 2 * 2 * 4


def test_zero_query_and_determinism(cuda_lib):
    cfg = wl.small_config(B=1, Hq=4, Hkv=2, L=300, window=8, pool=5, budget=40)
    Q, K, V = _inputs(cfg)
    a = gpu_compress(Q, K, V, window=8, pool=5, budget=40, n_cal=8, cap=44)
    b = gpu_compress(Q, K, V, window=8, pool=5, budget=40, n_cal=8, cap=44)
    for name in ("kept_idx", "K_kept", "V_kept", "O_c", "LSE_c", "C_q", "vote", "pooled"):
        np.testing.assert_array_equal(getattr(a, name), getattr(b, name), err_msg=name)
    ref, _ = compare_compress(a, Q, K, V, window=8, pool=5, budget=40, n_cal=8)
    z = np.zeros((1, 1, 4, 128), dtype=np.uint16)
    st = decode_steps_compare(a, ref, z, z[:, :, :2], z[:, :, :2], steps=1, append=False)
    assert st["applied"] == 0


def test_invalid_arguments_have_no_effect(cuda_lib):
    cd = cuda_lib
    cfg = wl.small_config()
    Q, K, V = _inputs(cfg)
    good = dict(B=1, Hq=4, Hkv=2, L=300, window=8, pool=5, budget=40, n_cal=1, cap=40)
    st = cd.alloc_layer_state(cd.make_params(**good))
    dQ, dK, dV = to_dev(Q), to_dev(K), to_dev(V)
    st.kept_idx.fill_(-7)

    def call(**kw):
        p = cd.make_params(**{**good, **kw})
        return cd.calidrop_compress(p, dQ, dK, dV, None, st.kept_idx, st.K_kept, st.V_kept, st.O_c, st.LSE_c,
                                    st.C_q, st.ws_compress, check=False)

    assert call(budget=8) == cd.INVALID_ARG          # budget <= window < L
    assert call(pool=4) == cd.INVALID_ARG
    assert call(n_cal=9) == cd.INVALID_ARG
    assert call(cap=10) == cd.INVALID_ARG
    assert call(D=64) == cd.UNSUPPORTED
    assert call(Hq=18, Hkv=2) == cd.UNSUPPORTED      # G = 9
    assert call(Hq=5) == cd.INVALID_ARG
    p = cd.make_params(**good)
    assert cd.calidrop_compress(p, None, dK, dV, None, st.kept_idx, st.K_kept, st.V_kept, st.O_c, st.LSE_c,
                                st.C_q, st.ws_compress, check=False) == cd.INVALID_ARG
    assert cd.calidrop_compress(p, dQ.view(torch.uint8)[2:].view(torch.bfloat16), dK, dV, None, st.kept_idx,
                                st.K_kept, st.V_kept, st.O_c, st.LSE_c, st.C_q, st.ws_compress,
                                check=False) == cd.INVALID_ARG
    assert cd.calidrop_compress(p, dQ, dK, dV, None, st.kept_idx, st.K_kept, st.V_kept, st.O_c, st.LSE_c,
                                st.C_q, st.ws_compress[:256], check=False) == cd.WORKSPACE_TOO_SMALL
    torch.cuda.synchronize()
    assert torch.all(st.kept_idx == -7)              # failed calls launched nothing
    out = torch.empty((1, 4, 128), dtype=torch.bfloat16, device="cuda")
    dq = to_dev(np.zeros((1, 4, 128), np.uint16))
    assert cd.calidrop_decode(p, dq, None, None, st.K_kept, st.V_kept, 0, st.O_c, st.LSE_c, st.C_q, out, None,
                              None, st.ws_decode, check=False) == cd.INVALID_ARG     # empty cache
    assert cd.calidrop_decode(p, dq, None, None, st.K_kept, st.V_kept, 41, st.O_c, st.LSE_c, st.C_q, out, None,
                              None, st.ws_decode, check=False) == cd.INVALID_ARG     # beyond cap
    assert "invalid" in cd.status_string(cd.INVALID_ARG)


def test_binding_refuses_what_it_cannot_pass_on(cuda_lib):
    """The native marshalling: tensors, addresses, None and integers of any integer type go through; strided
    tensors, wrong counts and other objects raise before anything is enqueued."""
    cd = cuda_lib
    cfg = wl.small_config()
    Q, K, V = _inputs(cfg)
    g = gpu_compress(Q, K, V, window=8, pool=5, budget=40, n_cal=1, cap=42)
    p, st = g.p, g.st
    q = to_dev(wl.gen_decode_inputs(cfg, Q, steps=1)[0][0])
    out = torch.full((1, 4, 128), 7.0, dtype=torch.bfloat16, device="cuda")

    def call(qq=q, kv_len=40, oo=out, ws=st.ws_decode):
        return cd.calidrop_decode(p, qq, None, None, st.K_kept, st.V_kept, kv_len, st.O_c, st.LSE_c, st.C_q, oo, None, None,
                                  ws)

    launches = cd.calidrop_launch_count()
    with pytest.raises(AssertionError):
        call(qq=torch.empty((1, 4, 256), dtype=torch.bfloat16, device="cuda")[:, :, ::2])
    with pytest.raises(TypeError):
        call(qq="q")
    with pytest.raises(TypeError):
        call(ws=None)
    with pytest.raises(OverflowError):
        call(kv_len=1 << 40)
    with pytest.raises(cd.CalidropError):
        call(qq=None)
    with pytest.raises(TypeError):
        cd.native().decode(p, q)
    assert cd.calidrop_launch_count() == launches and torch.all(out == 7.0)
    call(kv_len=np.int32(40))
    want = out.clone()
    out.zero_()
    call(qq=q.data_ptr(), oo=out.data_ptr())
    assert torch.equal(out, want)


def test_batched_layers_match_single_layer_calls(cuda_lib):
    cd = cuda_lib
    cfg = wl.small_config(B=2, Hq=4, Hkv=2, L=260, window=8, pool=5, budget=40, layers=3)
    layers, singles = [], []
    out_b = []
    for layer in range(3):
        Q, K, V = _inputs(cfg, layer)
        g = gpu_compress(Q, K, V, window=8, pool=5, budget=40, n_cal=4, cap=42)
        q, kn, vn = wl.gen_decode_inputs(cfg, Q, layer, steps=1)
        dq, dk, dv = to_dev(q[0]), to_dev(kn[0]), to_dev(vn[0])
        Kb, Vb = g.st.K_kept.clone(), g.st.V_kept.clone()
        ob = torch.empty((2, 4, 128), dtype=torch.bfloat16, device="cuda")
        lb = torch.empty((2, 4), dtype=torch.float32, device="cuda")
        fb = torch.empty((2, 4), dtype=torch.uint8, device="cuda")
        layers.append(dict(q=dq, k_new=dk, v_new=dv, K_kept=Kb, V_kept=Vb, O_c=g.st.O_c, LSE_c=g.st.LSE_c,
                           C_q=g.st.C_q, out=ob, lse_out=lb, flags=fb))
        out_b.append((ob, lb, fb, Kb, Vb))
        os_ = torch.empty_like(ob); ls = torch.empty_like(lb); fs = torch.empty_like(fb)
        cd.calidrop_decode(g.p, dq, dk, dv, g.st.K_kept, g.st.V_kept, 40, g.st.O_c, g.st.LSE_c, g.st.C_q, os_, ls,
                           fs, g.st.ws_decode)
        singles.append((os_, ls, fs, g.st.K_kept, g.st.V_kept))
        p = g.p
    ws = torch.zeros((cd.calidrop_decode_workspace_bytes(p, 42) * 3,), dtype=torch.uint8, device="cuda")
    cd.calidrop_decode_batched(p, cd.make_decode_layers(layers), 40, ws)
    torch.cuda.synchronize()
    for (ob, lb, fb, Kb, Vb), (os_, ls, fs, Ks, Vs) in zip(out_b, singles):
        # the split factor differs between the two launches, so outputs agree to rounding only
        assert torch.allclose(ob.float(), os_.float(), atol=2e-2)
        assert torch.allclose(lb, ls, atol=1e-4)
        assert torch.equal(fb, fs)
        assert torch.equal(Kb, Ks) and torch.equal(Vb, Vs)


# ---------------------------------------------------------------- the benchmark configurations
def _run_config_full(cfg, n_cal, steps):
    Q, K, V = _inputs(cfg)
    g = gpu_compress(Q, K, V, window=cfg.window, pool=cfg.pool, budget=cfg.budget, n_cal=n_cal,
                     cap=cfg.budget + steps)
    ref, swaps = compare_compress(g, Q, K, V, window=cfg.window, pool=cfg.pool, budget=cfg.budget, n_cal=n_cal)
    q, kn, vn = wl.gen_decode_inputs(cfg, Q, steps=steps)
    st = decode_steps_compare(g, ref, q, kn, vn, steps=steps)
    return swaps, st


@pytest.mark.parametrize("n_cal", [1, 32])
def test_config1_full(cuda_lib, n_cal):
    cfg = wl.CONFIGS[1]
    swaps, st = _run_config_full(cfg, n_cal, cfg.steps)
    assert st["applied"] > 0.5 * st["total"]      # cos-sim ~0.9 > theta2: calibration is exercised


@pytest.mark.parametrize("n_cal", [1, 32])
def test_config2_full(cuda_lib, n_cal):
    cfg = wl.CONFIGS[2]
    swaps, st = _run_config_full(cfg, n_cal, cfg.steps)
    assert st["applied"] > 0.5 * st["total"]


def _sampled_units_check(cfg, layer, n_cal, units, steps, step_ids, compress_units=None):
    """Full-size GPU run through the C-ABI.  The oracle evaluates compress-and-calibrate on
    `compress_units` (default: `units`) and the decode steps `step_ids` on `units`; the sampled units
    go to the oracle as one batch, so that its loop over units runs on all host cores.
    Returns (number of heads that applied the calibration, number that did not) over the checked steps."""
    Q, K, V = _inputs(cfg, layer)
    T = steps
    g = gpu_compress(Q, K, V, window=cfg.window, pool=cfg.pool, budget=cfg.budget, n_cal=n_cal,
                     cap=cfg.budget + T)
    G = cfg.G
    q, kn, vn = wl.gen_decode_inputs(cfg, Q, layer, steps=T)
    # GPU decode over all steps, recording the sampled steps' outputs
    from paper_2507_19906_b200 import binding as cd
    p, st = g.p, g.st
    out = torch.empty((p.B, p.Hq, p.D), dtype=torch.bfloat16, device="cuda")
    lse = torch.empty((p.B, p.Hq), dtype=torch.float32, device="cuda")
    flags = torch.empty((p.B, p.Hq), dtype=torch.uint8, device="cuda")
    rec = {}
    for t in range(T):
        cd.calidrop_decode(p, to_dev(q[t]), to_dev(kn[t]), to_dev(vn[t]), st.K_kept, st.V_kept, cfg.budget + t,
                           st.O_c, st.LSE_c, st.C_q, out, lse, flags, st.ws_decode)
        if t in step_ids:
            torch.cuda.synchronize()
            rec[t] = (wl.bf16_bits_to_f64(to_bits(out)), lse.cpu().numpy(), flags.cpu().numpy())
    torch.cuda.synchronize()
    off = cd.calidrop_decode_workspace_status_offset(p)
    assert int(st.ws_decode[off:off + 4].view(torch.int32).item()) == 0, "a wait of the decode kernel ran out"

    # the sampled units as a batch of single-kv-head problems: [n, G, W, D] queries, [n, 1, L, D] keys/values
    cu = list(compress_units if compress_units is not None else units)
    assert set(units) <= set(cu)
    hsl = lambda h: slice(h * G, (h + 1) * G)
    Qs = np.ascontiguousarray(np.stack([Q[b, hsl(h)] for b, h in cu]))
    Ks = np.ascontiguousarray(np.stack([K[b, h:h + 1] for b, h in cu]))
    Vs = np.ascontiguousarray(np.stack([V[b, h:h + 1] for b, h in cu]))
    sub = type("R", (), {})()
    sub.kept_idx = np.stack([g.kept_idx[b, h:h + 1] for b, h in cu])
    sub.K_kept = np.stack([g.K_kept[b, h:h + 1] for b, h in cu])
    sub.V_kept = np.stack([g.V_kept[b, h:h + 1] for b, h in cu])
    sub.O_c = np.stack([g.O_c[b, hsl(h)] for b, h in cu])
    sub.LSE_c = np.stack([g.LSE_c[b, hsl(h)] for b, h in cu])
    sub.C_q = np.stack([g.C_q[b, hsl(h)] for b, h in cu])
    sub.n_kept, sub.cap = g.n_kept, g.cap
    ref, swaps = compare_compress(sub, Qs, Ks, Vs, window=cfg.window, pool=cfg.pool, budget=cfg.budget, n_cal=n_cal)

    applied = not_applied = 0
    for (b, h) in units:
        i = cu.index((b, h))
        hs = hsl(h)
        Kk, Vk = ref.K_kept[i:i + 1].copy(), ref.V_kept[i:i + 1].copy()
        Oc, Lc, Cq = ref.O_c[i:i + 1], ref.LSE_c[i:i + 1], ref.C_q[i:i + 1]
        for t in range(T):
            qs = np.ascontiguousarray(q[t, b:b + 1, hs])
            kns = np.ascontiguousarray(kn[t, b:b + 1, h:h + 1])
            vns = np.ascontiguousarray(vn[t, b:b + 1, h:h + 1])
            if t not in step_ids:
                Kk[0, 0, cfg.budget + t], Vk[0, 0, cfg.budget + t] = kns[0, 0], vns[0, 0]
                continue
            o = oracle.decode(qs, kns, vns, Kk, Vk, cfg.budget + t, Oc, Lc, Cq)
            gout, glse, gfl = rec[t]
            gf = gfl[b, hs]
            if not np.array_equal(gf, o.flags[0]):
                fc = (gf >> 2).astype(np.int32)[None]
                fa = (gf & 1).astype(np.int32)[None]
                for k in np.nonzero(gf != o.flags[0])[0]:
                    rho = o.rho[0, k]
                    assert abs(rho[gf[k] >> 2] - rho.max()) < 1e-4
                    assert (gf[k] & 1) == (o.flags[0, k] & 1) or abs(rho.max() - 0.85) < 1e-3
                o = oracle.decode(qs, None, None, Kk, Vk, cfg.budget + t + 1, Oc, Lc, Cq,
                                  force_c=fc, force_apply=fa)
            assert_close_out(gout[b, hs], o.out[0], f"layer {layer} unit ({b},{h}) step {t}")
            assert_close_lse(glse[b, hs], o.lse[0], f"layer {layer} unit ({b},{h}) step {t} lse")
            applied += int((gf & 1).sum())
            not_applied += int((1 - (gf & 1)).sum())
    return applied, not_applied


# ---------------------------------------------------------------- the configurations at full size
def test_config3_every_unit_and_every_decode_step(cuda_lib):
    """Config 3 as benchmarked (n_cal = W = 64): compress-and-calibrate of all 32 units against the
    oracle, and all 128 decode steps on four units (one per batch element)."""
    cfg = wl.CONFIGS[3]
    every = [(b, h) for b in range(cfg.B) for h in range(cfg.Hkv)]
    applied, _ = _sampled_units_check(cfg, 0, n_cal=64, units=[(0, 0), (1, 3), (2, 6), (3, 7)], steps=cfg.steps,
                                      step_ids=set(range(cfg.steps)), compress_units=every)
    assert applied > 0


def test_config4_every_layer(cuda_lib):
    """Config 4: each of the 32 layers at full size on the GPU, two units per layer against the oracle
    (the units move with the layer so that every batch element and kv head is visited)."""
    cfg = wl.CONFIGS[4]
    for layer in range(cfg.layers):
        units = [(layer % cfg.B, (layer // 4) % cfg.Hkv), ((layer + 3) % cfg.B, (layer + 5) % cfg.Hkv)]
        _sampled_units_check(cfg, layer, n_cal=32, units=units, steps=4, step_ids={0, 3})


def test_config5_every_unit_and_the_drift_across_the_gate(cuda_lib):
    """Config 5: all four units of the 131072-token prompt, and decode steps spread over the whole run
    of 512: the query noise grows with the step, so early steps apply the calibration and late steps,
    past the point where the similarity falls below theta2, do not.  Both must occur."""
    cfg = wl.CONFIGS[5]
    every = [(0, h) for h in range(cfg.Hkv)]
    applied, not_applied = _sampled_units_check(cfg, 0, n_cal=64, units=every, steps=cfg.steps,
                                                step_ids={0, 100, 200, 300, 400, 480, 511})
    assert applied > 0 and not_applied > 0


def test_config3_sampled_units(cuda_lib):
    cfg = wl.CONFIGS[3]
    _sampled_units_check(cfg, 0, n_cal=64, units=[(0, 0), (3, 5)], steps=8, step_ids={0, 7})


def test_config3_sampled_units_last_query_only(cuda_lib):
    cfg = wl.CONFIGS[3]
    _sampled_units_check(cfg, 0, n_cal=1, units=[(1, 7)], steps=2, step_ids={1})


def test_config5_last_query_only(cuda_lib):
    cfg = wl.CONFIGS[5]
    _sampled_units_check(cfg, 0, n_cal=1, units=[(0, 2)], steps=4, step_ids={3})


# ---------------------------------------------------------------- decode on hand-built states
@pytest.mark.parametrize("B,Hq,Hkv,kv0,steps,n_cal", [
    (1, 4, 2, 0, 6, 3),       # the cache starts empty: the first step attends to its own row alone
    (2, 8, 2, 60, 8, 2),      # the appended row crosses the first 64-row slot boundary
    (1, 7, 1, 1020, 10, 5),   # ... and a 16-row block boundary deep in a slice
    (3, 8, 8, 250, 4, 1),     # 24 units: clusters of 4, slices of about 64 rows
    (1, 4, 1, 16500, 3, 2),   # one unit, 16500 rows: several clusters meet through the workspace
    (1, 8, 2, 40000, 2, 1),   # two units, 40000 rows each: several clusters per unit
])
def test_decode_ignores_cache_rows_beyond_kv_len(cuda_lib, B, Hq, Hkv, kv0, steps, n_cal):
    """The cache rows at and beyond kv_len belong to the caller and may hold anything; here they
    hold NaN bit patterns.  Every step must still match the oracle, which never reads them."""
    from paper_2507_19906_b200 import binding as cd
    rng = np.random.Generator(np.random.Philox(key=[77, B * 1000 + kv0]))
    D, cap = 128, max(kv0 + steps, 64)
    bits = lambda x: wl.f32_to_bf16_bits(np.ascontiguousarray(x, dtype=np.float32))
    budget = min(cap, max(kv0, 16))
    p = cd.make_params(B=B, Hq=Hq, Hkv=Hkv, L=budget + 64, window=8, pool=7, budget=budget, n_cal=n_cal, cap=cap)
    st = cd.alloc_layer_state(p)
    Kk = np.full((B, Hkv, cap, D), 0x7FC0, dtype=np.uint16)   # quiet NaN everywhere ...
    Vk = np.full((B, Hkv, cap, D), 0x7FC0, dtype=np.uint16)
    Kk[:, :, :kv0] = bits(rng.standard_normal((B, Hkv, kv0, D)))   # ... except the valid rows
    Vk[:, :, :kv0] = bits(rng.standard_normal((B, Hkv, kv0, D)))
    Cq = bits(rng.standard_normal((B, Hq, n_cal, D)))
    Oc = rng.standard_normal((B, Hq, n_cal, D)).astype(np.float32)
    Lc = (rng.standard_normal((B, Hq, n_cal)) + 3.0).astype(np.float32)
    st.K_kept.copy_(to_dev(Kk)); st.V_kept.copy_(to_dev(Vk)); st.C_q.copy_(to_dev(Cq))
    st.O_c.copy_(torch.from_numpy(Oc)); st.LSE_c.copy_(torch.from_numpy(Lc))
    out = torch.empty((B, Hq, D), dtype=torch.bfloat16, device="cuda")
    lse = torch.empty((B, Hq), dtype=torch.float32, device="cuda")
    flags = torch.empty((B, Hq), dtype=torch.uint8, device="cuda")
    p.theta1, p.theta2 = 0.7, -1.0                                  # always merge: O_c and LSE_c matter
    for t in range(steps):
        # queries close to a calibration query half of the time, so that both rows get chosen
        q = bits(wl.bf16_bits_to_f32(Cq[:, :, t % n_cal]) + 0.5 * rng.standard_normal((B, Hq, D)).astype(np.float32))
        kn, vn = bits(rng.standard_normal((B, Hkv, D))), bits(rng.standard_normal((B, Hkv, D)))
        cd.calidrop_decode(p, to_dev(q), to_dev(kn), to_dev(vn), st.K_kept, st.V_kept, kv0 + t, st.O_c, st.LSE_c,
                           st.C_q, out, lse, flags, st.ws_decode)
        torch.cuda.synchronize()
        o = oracle.decode(q, kn, vn, Kk, Vk, kv0 + t, Oc, Lc, Cq, theta1=0.7, theta2=-1.0)
        got = wl.bf16_bits_to_f64(to_bits(out))
        gf = flags.cpu().numpy()
        if not np.array_equal(gf >> 2, o.flags >> 2):
            # the chosen calibration row may differ only when the two similarities are within 1e-4;
            # the oracle is then re-evaluated under the GPU's choice
            force_c = np.full((B, Hq), -1, dtype=np.int32)
            for b, hq in zip(*np.nonzero((gf >> 2) != (o.flags >> 2))):
                gc, oc = int(gf[b, hq] >> 2), int(o.flags[b, hq] >> 2)
                assert abs(o.rho[b, hq, gc] - o.rho[b, hq, oc]) < 1e-4, "calibration row differs beyond a near-tie"
                force_c[b, hq] = gc
            o = oracle.decode(q, None, None, Kk, Vk, kv0 + t + 1, Oc, Lc, Cq, theta1=0.7, theta2=-1.0,
                              force_c=force_c)
        assert_close_out(got, o.out, f"step {t}")
        assert_close_lse(lse.cpu().numpy(), o.lse, f"step {t} lse")
        # the appended row reached the cache, bit for bit, and nothing else was written
        np.testing.assert_array_equal(to_bits(st.K_kept)[:, :, :kv0 + t + 1], Kk[:, :, :kv0 + t + 1])
        np.testing.assert_array_equal(to_bits(st.V_kept)[:, :, :kv0 + t + 1], Vk[:, :, :kv0 + t + 1])
        np.testing.assert_array_equal(to_bits(st.K_kept)[:, :, kv0 + t + 1:], Kk[:, :, kv0 + t + 1:])


@pytest.mark.parametrize("units,layers,G,kv,n_cal,layout", [
    # layout: CTAs of a cluster, clusters per unit, CTAs per SM
    (80, 2, 1, 64, 1, (1, 1, 2)),         # one calibration row, one whole slot and the appended row
    (80, 3, 4, 700, 33, (1, 1, 2)),       # 132 calibration rows, four of them in a second slot
    (20, 8, 3, 2100, 64, (1, 1, 2)),      # a long slice
    (80, 4, 8, 0, 64, (1, 1, 4)),         # the appended row alone
    (75, 5, 7, 32, 100, (1, 1, 4)),       # eleven slots of calibration rows, the last with 60; n_cal above 64
    (80, 4, 2, 1023, 16, (1, 1, 4)),      # the longest slice of this shape
    (80, 4, 2, 1024, 16, (1, 1, 1)),      # one more row: the wide ring, more CTAs than SMs
    (3, 1, 7, 4400, 5, (16, 1, 1)),       # five calibration rows over sixteen CTAs
    (1, 2, 8, 9001, 64, (16, 1, 1)),      # ... 64, in two layers
    (1, 2, 8, 17000, 64, (8, 5, 1)),      # several clusters of eight
    (16, 1, 4, 2100, 8, (4, 1, 1)),       # more clusters of eight than the GPU holds at once
    (4, 1, 4, 1199, 8, (16, 1, 1)),       # slices of 75 rows are launched as 80, of 150 as 160
    (12, 1, 4, 649, 8, (8, 1, 1)),        # ... of 82 as 96, of 163 as 176
    (1, 1, 8, 12449, 16, (16, 1, 1)),     # ... of 195 (on 64 CTAs) as 208
])
def test_decode_launch_shapes_against_fp32(cuda_lib, units, layers, G, kv, n_cal, layout):
    """Every shape that the launch rules choose between, at its edges, against the same step in fp32: outputs are bf16
    of values below about 2 (tolerances of the other parity tests); the calibration row is the one the query was
    drawn around, far from any tie."""
    cd = cuda_lib
    gen = torch.Generator(device="cuda").manual_seed(units * 7 + kv)
    rn = lambda *sh: torch.randn(sh, generator=gen, device="cuda")
    Hq, cap = units * G, kv + 3
    p = cd.make_params(B=1, Hq=Hq, Hkv=units, n_cal=n_cal, cap=cap)
    p.theta1, p.theta2 = 0.7, -1.0
    plan = cd.calidrop_decode_plan(p, layers, kv + 1)
    assert (plan.cluster_ctas, plan.clusters_per_unit, plan.ctas_per_sm) == layout
    bf = torch.bfloat16
    ins = []
    for i in range(layers):
        pick = torch.randint(n_cal, (1, Hq), generator=gen, device="cuda")
        C_q = rn(1, Hq, n_cal, 128).to(bf)
        q = (C_q.float().gather(2, pick[..., None, None].expand(-1, -1, 1, 128))[:, :, 0] + 0.3 * rn(1, Hq, 128)).to(bf)
        ins.append(dict(q=q, k_new=rn(1, units, 128).to(bf), v_new=rn(1, units, 128).to(bf),
                        K_kept=rn(1, units, cap, 128).to(bf), V_kept=rn(1, units, cap, 128).to(bf),
                        O_c=rn(1, Hq, n_cal, 128), LSE_c=rn(1, Hq, n_cal) + 6, C_q=C_q,
                        out=torch.empty((1, Hq, 128), dtype=bf, device="cuda"),
                        lse_out=torch.empty((1, Hq), device="cuda"),
                        flags=torch.empty((1, Hq), dtype=torch.uint8, device="cuda"), pick=pick))
    ws = torch.zeros((cd.calidrop_decode_workspace_bytes(p, cap) * layers,), dtype=torch.uint8, device="cuda")
    cd.calidrop_decode_batched(p, cd.make_decode_layers([{k: v for k, v in d.items() if k != "pick"} for d in ins]), kv, ws)
    torch.cuda.synchronize()
    off = cd.calidrop_decode_workspace_status_offset(p)
    assert int(ws[off:off + 4].view(torch.int32).item()) == 0
    for d in ins:
        assert torch.equal(d["K_kept"][:, :, kv], d["k_new"]) and torch.equal(d["V_kept"][:, :, kv], d["v_new"])
        if n_cal <= 64:
            assert torch.equal((d["flags"] >> 2).long(), d["pick"])
        K, V = (d[k][0, :, :kv + 1].float() for k in ("K_kept", "V_kept"))
        s = torch.einsum("ugd,utd->ugt", d["q"].float().view(units, G, 128).double(), K.double()) / 128 ** 0.5
        la = torch.logsumexp(s, -1)
        oa = torch.einsum("ugt,utd->ugd", torch.softmax(s, -1), V.double())
        lc = d["LSE_c"].gather(2, d["pick"][..., None])[..., 0].view(units, G).double()
        oc = d["O_c"].gather(2, d["pick"][..., None, None].expand(-1, -1, 1, 128)).view(units, G, 128).double()
        lse = torch.logaddexp(la, lc)
        want = torch.exp(la - lse)[..., None] * oa + torch.exp(lc - lse)[..., None] * oc
        assert (d["out"].double().view(units, G, 128) - want).abs().max() < 2e-2 * max(1.0, want.abs().max().item() / 2)
        assert (d["out"].double().view(units, G, 128) - want).abs().mean() < 2e-3
        assert (d["lse_out"].double().view(units, G) - lse).abs().max() < 1e-3


def test_batched_layers_with_several_clusters_per_unit(cuda_lib):
    """Two layers of one unit with 17000 cached rows in one launch: every (layer, unit) is split over
    several clusters that meet through the workspace, each layer with its own counters and partials.
    Checked against the oracle, twice on the same workspace (the counters must come back to zero)."""
    cd = cuda_lib
    rng = np.random.Generator(np.random.Philox(key=[91, 5]))
    B, Hq, Hkv, D, kv0, n_cal, NL = 1, 4, 1, 128, 17000, 2, 2
    cap = kv0 + 2
    bits = lambda x: wl.f32_to_bf16_bits(np.ascontiguousarray(x, dtype=np.float32))
    p = cd.make_params(B=B, Hq=Hq, Hkv=Hkv, L=kv0 + 64, window=8, pool=7, budget=kv0, n_cal=n_cal, cap=cap)
    p.theta1, p.theta2 = 0.7, -1.0
    assert cd.calidrop_decode_plan(p, NL, kv0 + 1).clusters_per_unit > 1
    ws = torch.zeros((cd.calidrop_decode_workspace_bytes(p, cap) * NL,), dtype=torch.uint8, device="cuda")
    host, layers = [], []
    for _ in range(NL):
        Kk = np.zeros((B, Hkv, cap, D), dtype=np.uint16); Vk = np.zeros_like(Kk)
        Kk[:, :, :kv0] = bits(rng.standard_normal((B, Hkv, kv0, D)))
        Vk[:, :, :kv0] = bits(rng.standard_normal((B, Hkv, kv0, D)))
        Cq = bits(rng.standard_normal((B, Hq, n_cal, D)))
        Oc = rng.standard_normal((B, Hq, n_cal, D)).astype(np.float32)
        Lc = (rng.standard_normal((B, Hq, n_cal)) + 9.0).astype(np.float32)
        dev = dict(K_kept=to_dev(Kk), V_kept=to_dev(Vk), C_q=to_dev(Cq), O_c=torch.from_numpy(Oc).cuda(),
                   LSE_c=torch.from_numpy(Lc).cuda(),
                   out=torch.empty((B, Hq, D), dtype=torch.bfloat16, device="cuda"),
                   lse_out=torch.empty((B, Hq), dtype=torch.float32, device="cuda"),
                   flags=torch.empty((B, Hq), dtype=torch.uint8, device="cuda"))
        host.append((Kk, Vk, Cq, Oc, Lc)); layers.append(dev)
    for t in range(2):
        step = []
        for dev, (Kk, Vk, Cq, Oc, Lc) in zip(layers, host):
            q = bits(wl.bf16_bits_to_f32(Cq[:, :, t % n_cal]) + 0.5 * rng.standard_normal((B, Hq, D)).astype(np.float32))
            kn, vn = bits(rng.standard_normal((B, Hkv, D))), bits(rng.standard_normal((B, Hkv, D)))
            dev.update(q=to_dev(q), k_new=to_dev(kn), v_new=to_dev(vn))
            step.append((q, kn, vn))
        cd.calidrop_decode_batched(p, cd.make_decode_layers(layers), kv0 + t, ws)
        torch.cuda.synchronize()
        off = cd.calidrop_decode_workspace_status_offset(p)
        assert int(ws[off:off + 4].view(torch.int32).item()) == 0
        for dev, (Kk, Vk, Cq, Oc, Lc), (q, kn, vn) in zip(layers, host, step):
            o = oracle.decode(q, kn, vn, Kk, Vk, kv0 + t, Oc, Lc, Cq, theta1=0.7, theta2=-1.0)
            same = (dev["flags"].cpu().numpy() >> 2) == (o.flags >> 2)
            assert same.all()
            assert_close_out(wl.bf16_bits_to_f64(to_bits(dev["out"])), o.out, f"step {t}")
            assert_close_lse(dev["lse_out"].cpu().numpy(), o.lse, f"step {t} lse")
            np.testing.assert_array_equal(to_bits(dev["K_kept"]), Kk)


# ---------------------------------------------------------------- a kept list chosen by the caller
def _streaming_indices(B, Hkv, L, budget, n_sink):
    """Index rule of a sink-plus-recent cache: the first n_sink rows and the most recent ones."""
    idx = np.concatenate([np.arange(n_sink), np.arange(L - (budget - n_sink), L)]).astype(np.int32)
    return np.broadcast_to(idx, (B, Hkv, budget)).copy()


@pytest.mark.parametrize("B,Hq,Hkv,L,W,budget,n_cal,rule,supply_lse", [
    (1, 4, 2, 700, 16, 96, 4, "streaming", False),
    (2, 8, 2, 1500, 32, 256, 32, "random", False),     # two 128-row calibration blocks per kv head
    (1, 7, 1, 3000, 64, 400, 64, "streaming", True),   # G = 7, row LSE supplied by the caller
])
def test_calibrate_with_a_supplied_kept_list(cuda_lib, B, Hq, Hkv, L, W, budget, n_cal, rule, supply_lse):
    cd = cuda_lib
    cfg = wl.small_config(B=B, Hq=Hq, Hkv=Hkv, L=L, window=W, pool=7, budget=budget, steps=3,
                          n_sink=4, n_heavy=max(1, L // 50))
    Q, K, V = _inputs(cfg)
    if rule == "streaming":
        kept = _streaming_indices(B, Hkv, L, budget, 32)
    else:
        rng = np.random.Generator(np.random.Philox(key=[5, L]))
        kept = np.stack([np.stack([np.sort(np.concatenate([
            rng.choice(L - W, size=budget - W, replace=False), np.arange(L - W, L)])).astype(np.int32)
            for _ in range(Hkv)]) for _ in range(B)])
    T = 3
    p = cd.make_params(B=B, Hq=Hq, Hkv=Hkv, L=L, window=W, pool=7, budget=budget, n_cal=n_cal, cap=budget + T)
    st = cd.alloc_layer_state(p)
    ref = oracle.calibrate_given_indices(Q, K, V, kept, n_cal=n_cal, cap=budget + T)
    lse = None
    if supply_lse:
        lse = torch.from_numpy(oracle.compress(Q, K, V, window=W, pool=7, budget=budget, n_cal=n_cal)
                               .row_lse.astype(np.float32)).cuda()
    cd.calidrop_calibrate(p, to_dev(Q), to_dev(K), to_dev(V), lse, torch.from_numpy(kept).cuda(), st.K_kept,
                          st.V_kept, st.O_c, st.LSE_c, st.C_q, st.ws_compress)
    torch.cuda.synchronize()
    lay = cd.calidrop_compress_workspace_layout(p)
    assert int(st.ws_compress[lay.status_offset:lay.status_offset + 4].view(torch.int32).item()) == 0
    np.testing.assert_array_equal(to_bits(st.K_kept)[:, :, :budget], ref.K_kept[:, :, :budget])
    np.testing.assert_array_equal(to_bits(st.V_kept)[:, :, :budget], ref.V_kept[:, :, :budget])
    np.testing.assert_array_equal(to_bits(st.C_q), ref.C_q)
    assert_close_lse(st.LSE_c.cpu().numpy(), ref.LSE_c, "LSE_c")
    assert_close_out(st.O_c.cpu().numpy(), ref.O_c, "O_c")
    # and the decode steps that follow use this state like any other
    from types import SimpleNamespace
    g = SimpleNamespace(st=st, p=p, n_kept=budget)
    q, kn, vn = wl.gen_decode_inputs(cfg, Q, steps=T)
    res = decode_steps_compare(g, ref, q, kn, vn, steps=T)
    assert res["total"] == T * B * Hq


# ---------------------------------------------------------------- the recompute branch (Algorithm 2, lines 3-8)
@pytest.mark.parametrize("units,L,W,budget", [
    (3, 8192 + 8, 8, 40),         # one slice of the index kernel, full
    (3, 8192 + 9, 8, 8000),       # one candidate in the second slice, most rows kept
    (1, 40000, 32, 64),           # five slices
    (1, 330000, 8, 16),           # a bitmap longer than the one built in shared memory
])
def test_evicted_list_at_the_edges_of_its_slices(cuda_lib, units, L, W, budget):
    """The complement of a caller's list, in any order and with entries twice or outside the prompt: those leave fewer
    kept rows, and the rows past the budgeted number of evicted ones are dropped."""
    cd = cuda_lib
    rng = np.random.Generator(np.random.Philox(key=[67, L]))
    kept = np.stack([rng.permutation(L - W)[:budget] for _ in range(units)]).astype(np.int32)
    kept[0, 0], kept[0, 1] = -5, L + 3
    kept[-1, 2] = kept[-1, 3]
    p = cd.make_params(B=1, Hq=units, Hkv=units, L=L, window=W, pool=1, budget=budget, n_cal=1, cap=budget)
    n_e = L - budget
    K = torch.arange(L, device="cuda").view(1, 1, L, 1).expand(1, units, L, 128).to(torch.bfloat16).contiguous()
    V = -K
    ws = torch.empty((cd.calidrop_compress_workspace_bytes(p),), dtype=torch.uint8, device="cuda")
    ev = torch.empty((1, units, n_e), dtype=torch.int32, device="cuda")
    K_e = torch.zeros((1, units, n_e, 128), dtype=torch.bfloat16, device="cuda")
    V_e = torch.zeros_like(K_e)
    cd.calidrop_gather_evicted(p, K, V, torch.from_numpy(kept[None]).cuda(), ev, K_e, V_e, ws)
    got = ev.cpu().numpy()[0]
    for u in range(units):
        want = np.setdiff1d(np.arange(L - W), kept[u])[:n_e]
        np.testing.assert_array_equal(got[u, :len(want)], want)
        assert (got[u, len(want):] == -1).all()
        rows = torch.from_numpy(want).cuda()
        assert torch.equal(K_e[0, u, :len(want)], K[0, u, rows]) and torch.equal(V_e[0, u, :len(want)], V[0, u, rows])
        assert not K_e[0, u, len(want):].any()


@pytest.mark.parametrize("units,G,n_evict,layout", [
    (160, 3, 300, (1, 1, 2)),     # two CTAs per SM
    (300, 1, 1, (1, 1, 4)),       # four: a single row
    (300, 2, 1024, (1, 1, 4)),    # ... the longest slice of this shape
    (300, 1, 1025, (1, 1, 1)),    # one more row: the wide ring, more CTAs than SMs
    (2, 8, 2000, (8, 1, 1)),      # clusters of eight at the most
])
def test_recalibrate_launch_shapes_against_fp64(cuda_lib, units, G, n_evict, layout):
    """Every shape that a recomputation takes: O_c within the tolerance of bf16 probabilities, the other rows untouched."""
    cd = cuda_lib
    gen = torch.Generator(device="cuda").manual_seed(units + n_evict)
    rn = lambda *sh: torch.randn(sh, generator=gen, device="cuda")
    Hq, n_cal, slot = units * G, 3, 1
    p = cd.make_params(B=1, Hq=Hq, Hkv=units, n_cal=n_cal, cap=1)
    plan = cd.calidrop_decode_plan(p, 1, n_evict, True)
    assert (plan.cluster_ctas, plan.clusters_per_unit, plan.ctas_per_sm) == layout
    q, K, V = (rn(*sh).to(torch.bfloat16) for sh in ((1, Hq, 128), (1, units, n_evict, 128), (1, units, n_evict, 128)))
    O_c, LSE_c, C_q = rn(1, Hq, n_cal, 128), rn(1, Hq, n_cal), rn(1, Hq, n_cal, 128).to(torch.bfloat16)
    before = [t.clone() for t in (O_c, LSE_c, C_q)]
    ws = torch.zeros((cd.calidrop_decode_workspace_bytes(p, n_evict),), dtype=torch.uint8, device="cuda")
    cd.calidrop_recalibrate(p, q, K, V, n_evict, slot, O_c, LSE_c, C_q, ws)
    off = cd.calidrop_decode_workspace_status_offset(p)
    assert int(ws[off:off + 4].view(torch.int32).item()) == 0
    s = torch.einsum("ugd,utd->ugt", q.view(units, G, 128).double(), K[0].double()) / 128 ** 0.5
    want = torch.einsum("ugt,utd->ugd", torch.softmax(s, -1), V[0].double()).view(1, Hq, 128)
    assert (O_c[:, :, slot].double() - want).abs().max() < 2e-2 and (O_c[:, :, slot].double() - want).abs().mean() < 2e-3
    assert (LSE_c[:, :, slot].double() - torch.logsumexp(s, -1).view(1, Hq)).abs().max() < 1e-3
    assert torch.equal(C_q[:, :, slot], q)
    for got, was in zip((O_c, LSE_c, C_q), before):
        assert torch.equal(got[:, :, ::2], was[:, :, ::2])


@pytest.mark.parametrize("units,lengths", [
    (160, (900, 576, 900, 577, 300, 592)),   # a CTA to a unit: slices of up to 576 rows come by a copy per half, longer ones by one
    (4, (16000, 2000, 16000)),               # clusters
])
def test_slices_of_changing_length_over_the_same_buffers(cuda_lib, units, lengths):
    """Short and long slices are brought by different copies, each with descriptors of its own, also where steps and recomputations
    of either kind read the same buffers with the same capacity in turn.  Without a calibration applied both compute attention."""
    cd = cuda_lib
    gen = torch.Generator(device="cuda").manual_seed(units)
    rn = lambda *sh: torch.randn(sh, generator=gen, device="cuda")
    cap = max(lengths)
    p = cd.make_params(B=1, Hq=units, Hkv=units, n_cal=1, cap=cap, theta2=2.0)
    q, C_q = rn(1, units, 128).to(torch.bfloat16), rn(1, units, 1, 128).to(torch.bfloat16)
    K, V = (rn(1, units, cap, 128).to(torch.bfloat16) for _ in range(2))
    O_c, LSE_c = rn(1, units, 1, 128), rn(1, units, 1)
    out, lse = torch.empty((1, units, 128), dtype=torch.bfloat16, device="cuda"), torch.empty((1, units), device="cuda")
    ws = torch.zeros((cd.calidrop_decode_workspace_bytes(p, cap),), dtype=torch.uint8, device="cuda")
    s = torch.einsum("ud,utd->ut", q[0].double(), K[0].double()) / 128 ** 0.5
    off = cd.calidrop_decode_workspace_status_offset(p)
    for n in lengths:
        want, want_lse = torch.einsum("ut,utd->ud", torch.softmax(s[:, :n], -1), V[0, :, :n].double()), torch.logsumexp(s[:, :n], -1)
        out.zero_(), lse.zero_(), O_c.zero_(), LSE_c.zero_()
        cd.calidrop_decode(p, q, None, None, K, V, n, O_c, LSE_c, C_q, out, lse, None, ws)
        results = [(out[0], lse[0])]
        if n == cap:   # the same buffers as evicted rows
            cd.calidrop_recalibrate(p, q, K, V, n, 0, O_c, LSE_c, C_q, ws)
            results.append((O_c[0, :, 0], LSE_c[0, :, 0]))
        assert int(ws[off:off + 4].view(torch.int32).item()) == 0
        for o, l in results:
            assert (o.double() - want).abs().max() < 2e-2 and (o.double() - want).abs().mean() < 2e-3, n
            assert (l.double() - want_lse).abs().max() < 1e-3, n


@pytest.mark.parametrize("B,Hq,Hkv,L,W,budget,n_cal,slot", [
    (1, 4, 2, 600, 16, 80, 1, 0),          # the paper's single calibration query
    (2, 8, 2, 1500, 32, 256, 4, 2),        # G = 4, one of four rows rewritten
    (1, 7, 1, 20000, 64, 2048, 64, 63),    # one unit, 17952 evicted rows: several clusters of eight
])
def test_gather_evicted_and_recalibrate(cuda_lib, B, Hq, Hkv, L, W, budget, n_cal, slot):
    cd = cuda_lib
    cfg = wl.small_config(B=B, Hq=Hq, Hkv=Hkv, L=L, window=W, pool=7, budget=budget, steps=2,
                          n_sink=4, n_heavy=max(1, L // 50))
    Q, K, V = _inputs(cfg)
    g = gpu_compress(Q, K, V, window=W, pool=7, budget=budget, n_cal=n_cal, cap=budget + 2, keep_inputs=True)
    n_e = L - budget
    ev_idx = torch.empty((B, Hkv, n_e), dtype=torch.int32, device="cuda")
    K_e = torch.empty((B, Hkv, n_e, 128), dtype=torch.bfloat16, device="cuda")
    V_e = torch.empty_like(K_e)
    cd.calidrop_gather_evicted(g.p, g.dK, g.dV, g.st.kept_idx, ev_idx, K_e, V_e, g.st.ws_compress)
    torch.cuda.synchronize()
    ev = ev_idx.cpu().numpy()
    for b in range(B):
        for h in range(Hkv):
            want = np.setdiff1d(np.arange(L - W), g.kept_idx[b, h])     # ascending complement among candidates
            np.testing.assert_array_equal(ev[b, h], want)
            np.testing.assert_array_equal(to_bits(K_e)[b, h], K[b, h][want])
            np.testing.assert_array_equal(to_bits(V_e)[b, h], V[b, h][want])
    # a query far from every calibration query, as in the branch's condition
    rng = np.random.Generator(np.random.Philox(key=[11, L]))
    q = wl.f32_to_bf16_bits(rng.standard_normal((B, Hq, 128)).astype(np.float32))
    O_before, L_before, C_before = g.st.O_c.clone(), g.st.LSE_c.clone(), g.st.C_q.clone()
    cd.calidrop_recalibrate(g.p, to_dev(q), K_e, V_e, n_e, slot, g.st.O_c, g.st.LSE_c, g.st.C_q, g.st.ws_decode)
    torch.cuda.synchronize()
    off = cd.calidrop_decode_workspace_status_offset(g.p)
    assert int(g.st.ws_decode[off:off + 4].view(torch.int32).item()) == 0
    G = Hq // Hkv
    for b in range(B):
        for hq in range(Hq):
            h = hq // G
            o, l = oracle.full_attention(q[b, hq][None], K[b, h][ev[b, h]], V[b, h][ev[b, h]])
            assert_close_out(g.st.O_c[b, hq, slot].cpu().numpy(), o[0], "recomputed O_c")
            assert abs(float(g.st.LSE_c[b, hq, slot]) - l[0]) < 1e-3
    np.testing.assert_array_equal(to_bits(g.st.C_q)[:, :, slot], q)
    keep = [c for c in range(n_cal) if c != slot]                      # the other rows are untouched
    assert torch.equal(g.st.O_c[:, :, keep], O_before[:, :, keep])
    assert torch.equal(g.st.LSE_c[:, :, keep], L_before[:, :, keep])
    assert torch.equal(g.st.C_q[:, :, keep], C_before[:, :, keep])
    # the repeated decode step now finds rho = 1 with the new row and merges: the result is the
    # attention of q over the kept and the evicted rows together, i.e. over the whole prompt
    out = torch.empty((B, Hq, 128), dtype=torch.bfloat16, device="cuda")
    flags = torch.empty((B, Hq), dtype=torch.uint8, device="cuda")
    cd.calidrop_decode(g.p, to_dev(q), None, None, g.st.K_kept, g.st.V_kept, budget, g.st.O_c, g.st.LSE_c, g.st.C_q,
                       out, None, flags, g.st.ws_decode)
    torch.cuda.synchronize()
    f = flags.cpu().numpy()
    assert np.all(f & 1 == 1) and np.all(f & 2 == 0)
    got = wl.bf16_bits_to_f64(to_bits(out))
    for b in range(B):
        for hq in range(Hq):
            o, _ = oracle.full_attention(q[b, hq][None], K[b, hq // G], V[b, hq // G])
            assert_close_out(got[b, hq], o[0], "decode after the recompute vs attention over the whole prompt")


def test_offload_and_reload_of_the_evicted_rows_beside_decode(cuda_lib):
    """Algorithm 1 line 4 / Algorithm 2 line 4: the compacted evicted rows go to page-locked host
    memory on a copy stream and come back on it, bit for bit, while decode steps run on the compute
    stream; the decode outputs are the same as without the transfer, and a recompute from the
    reloaded rows equals one from the rows that never left."""
    cd = cuda_lib
    B, Hq, Hkv, L, W, budget, n_cal = 2, 8, 2, 6000, 32, 512, 32
    cfg = wl.small_config(B=B, Hq=Hq, Hkv=Hkv, L=L, window=W, pool=7, budget=budget, steps=6, n_sink=4, n_heavy=100)
    Q, K, V = _inputs(cfg)
    T = 6
    g = gpu_compress(Q, K, V, window=W, pool=7, budget=budget, n_cal=n_cal, cap=budget + T, keep_inputs=True)
    p, st = g.p, g.st
    n_e = L - budget
    ev_idx = torch.empty((B, Hkv, n_e), dtype=torch.int32, device="cuda")
    K_e = torch.empty((B, Hkv, n_e, 128), dtype=torch.bfloat16, device="cuda")
    V_e = torch.empty_like(K_e)
    K_h = torch.empty(K_e.shape, dtype=torch.bfloat16).pin_memory()
    V_h = torch.empty(V_e.shape, dtype=torch.bfloat16).pin_memory()
    main, side = torch.cuda.current_stream(), torch.cuda.Stream()
    gathered, offloaded, reloaded = torch.cuda.Event(), torch.cuda.Event(), torch.cuda.Event()
    cd.calidrop_gather_evicted(p, g.dK, g.dV, st.kept_idx, ev_idx, K_e, V_e, st.ws_compress)
    gathered.record(main)
    offloaded.record(side); reloaded.record(side)          # (creates the handles; they are recorded again below)
    cd.calidrop_offload_evicted(p, n_e, K_e, V_e, K_h, V_h, side, wait_event=gathered, done_event=offloaded)
    offloaded.synchronize()
    K_ref, V_ref = K_e.clone(), V_e.clone()
    assert torch.equal(K_h, K_ref.cpu()) and torch.equal(V_h, V_ref.cpu())
    # decode steps without any transfer, on copies of the cache
    q, kn, vn = wl.gen_decode_inputs(cfg, Q, steps=T)
    dq, dk, dv = [to_dev(x) for x in q], [to_dev(x) for x in kn], [to_dev(x) for x in vn]

    def run_steps(Kc, Vc):
        outs = []
        for t in range(T):
            o = torch.empty((B, Hq, 128), dtype=torch.bfloat16, device="cuda")
            cd.calidrop_decode(p, dq[t], dk[t], dv[t], Kc, Vc, budget + t, st.O_c, st.LSE_c, st.C_q, o, None, None,
                               st.ws_decode)
            outs.append(o)
        return outs

    quiet = run_steps(st.K_kept.clone(), st.V_kept.clone())
    torch.cuda.synchronize()
    # the device copy is dropped (overwritten), then reloaded on the side stream while decode runs
    K_e.zero_(); V_e.zero_()
    torch.cuda.synchronize()
    cd.calidrop_reload_evicted(p, n_e, K_h, V_h, K_e, V_e, side, wait_event=None, done_event=reloaded)
    busy = run_steps(st.K_kept.clone(), st.V_kept.clone())
    main.wait_event(reloaded)                              # the compute stream may read the rows from here on
    assert torch.equal(K_e, K_ref) and torch.equal(V_e, V_ref)
    for a, b in zip(quiet, busy):
        assert torch.equal(a, b)
    off = cd.calidrop_decode_workspace_status_offset(p)
    assert int(st.ws_decode[off:off + 4].view(torch.int32).item()) == 0
    # a recompute from the reloaded rows
    rng = np.random.Generator(np.random.Philox(key=[12, L]))
    qr = wl.f32_to_bf16_bits(rng.standard_normal((B, Hq, 128)).astype(np.float32))
    cd.calidrop_recalibrate(p, to_dev(qr), K_e, V_e, n_e, 5, st.O_c, st.LSE_c, st.C_q, st.ws_decode)
    torch.cuda.synchronize()
    ev = ev_idx.cpu().numpy()
    for b in range(B):
        for hq in range(Hq):
            h = hq // (Hq // Hkv)
            o, l = oracle.full_attention(qr[b, hq][None], K[b, h][ev[b, h]], V[b, h][ev[b, h]])
            assert_close_out(st.O_c[b, hq, 5].cpu().numpy(), o[0], "O_c recomputed from the reloaded rows")
            assert abs(float(st.LSE_c[b, hq, 5]) - l[0]) < 1e-3
    # argument checks
    assert cd.calidrop_offload_evicted(p, 0, K_e, V_e, K_h, V_h, side, check=False) == cd.INVALID_ARG
    assert cd.calidrop_reload_evicted(p, n_e, None, V_h, K_e, V_e, side, check=False) == cd.INVALID_ARG


def test_streaming_and_h2o_kept_lists_from_the_library_feed_the_calibration(cuda_lib):
    """The paper applies CaliDrop on top of StreamingLLM and H2O too (Sections 4.1.2-4.1.3): their kept
    lists, written on the device by the library, equal the oracle's, and calidrop_calibrate on them
    matches the oracle's calibration over the rows those rules evict."""
    cd = cuda_lib
    B, Hq, Hkv, L, W, budget, n_cal = 2, 4, 2, 700, 16, 128, 4
    G = Hq // Hkv
    cfg = wl.small_config(B=B, Hq=Hq, Hkv=Hkv, L=L, window=W, pool=1, budget=budget, steps=2, n_sink=4, n_heavy=14)
    Q, K, V = _inputs(cfg)
    p = cd.make_params(B=B, Hq=Hq, Hkv=Hkv, L=L, window=W, pool=1, budget=budget, n_cal=n_cal, cap=budget + 2)
    st = cd.alloc_layer_state(p)
    dQ, dK, dV = to_dev(Q), to_dev(K), to_dev(V)
    # H2O's accumulated attention needs every prompt query: a seeded full-query tensor whose last W rows are Q_obs
    rng = np.random.Generator(np.random.Philox(key=[31, 7]))
    scores = np.zeros((B, Hkv, L), dtype=np.float32)
    for b in range(B):
        for h in range(Hkv):
            Qfull = wl.f32_to_bf16_bits(rng.standard_normal((G, L, 128)).astype(np.float32))
            Qfull[:, L - W:] = Q[b, h * G:(h + 1) * G]
            scores[b, h] = oracle.accumulated_attention(Qfull, K[b, h]).astype(np.float32)
    lists = {}
    cd.calidrop_select_streaming(p, 32, st.kept_idx)
    torch.cuda.synchronize()
    lists["streaming"] = st.kept_idx.cpu().numpy().copy()
    np.testing.assert_array_equal(lists["streaming"], np.broadcast_to(oracle.streaming_indices(L, budget, 32), (B, Hkv, budget)))
    cd.calidrop_select_from_scores(p, torch.from_numpy(scores).cuda(), budget // 2, st.kept_idx, st.ws_compress)
    torch.cuda.synchronize()
    lists["h2o"] = st.kept_idx.cpu().numpy().copy()
    for b in range(B):
        for h in range(Hkv):
            # fp32 scores on both sides: the order is the same bit for bit
            np.testing.assert_array_equal(lists["h2o"][b, h], oracle.select_from_scores(scores[b, h], tail=budget // 2, budget=budget))
    for name, kept in lists.items():
        st.kept_idx.copy_(torch.from_numpy(kept))
        cd.calidrop_calibrate(p, dQ, dK, dV, None, st.kept_idx, st.K_kept, st.V_kept, st.O_c, st.LSE_c, st.C_q,
                              st.ws_compress)
        torch.cuda.synchronize()
        ref = oracle.calibrate_given_indices(Q, K, V, kept, n_cal=n_cal, cap=budget + 2)
        np.testing.assert_array_equal(to_bits(st.K_kept)[:, :, :budget], ref.K_kept[:, :, :budget])
        assert_close_lse(st.LSE_c.cpu().numpy(), ref.LSE_c, f"{name}: LSE_c")
        assert_close_out(st.O_c.cpu().numpy(), ref.O_c, f"{name}: O_c")
    # argument checks
    assert cd.calidrop_select_streaming(p, budget, st.kept_idx, check=False) == cd.INVALID_ARG
    assert cd.calidrop_select_from_scores(p, torch.from_numpy(scores).cuda(), W - 1, st.kept_idx, st.ws_compress,
                                          check=False) == cd.INVALID_ARG


@pytest.mark.parametrize("B,Hq,Hkv,L", [(1, 4, 2, 333), (2, 6, 2, 700), (1, 8, 1, 1100)])
def test_h2o_accumulated_scores_from_the_library(cuda_lib, B, Hq, Hkv, L):
    """H2O's importance measure (Section 4.1.2): the column sums of the causal attention of every prompt
    query, per kv head, computed by the library from Q and K, against the oracle's definition; the kept
    list that the library then selects from ITS scores equals the oracle's list from the oracle's scores
    up to swaps of rows whose oracle scores are closer than the fp32 arithmetic resolves."""
    cd = cuda_lib
    G, W, budget = Hq // Hkv, 16, 128
    rng = np.random.Generator(np.random.Philox(key=[41, L]))
    Qf = wl.f32_to_bf16_bits(rng.standard_normal((B, Hq, L, 128)).astype(np.float32))
    Kb = wl.f32_to_bf16_bits(rng.standard_normal((B, Hkv, L, 128)).astype(np.float32))
    Kb[:, :, ::37] = wl.f32_to_bf16_bits(2.5 * wl.bf16_bits_to_f32(Kb[:, :, ::37]))   # some heavy hitters
    p = cd.make_params(B=B, Hq=Hq, Hkv=Hkv, L=L, window=W, pool=1, budget=budget, n_cal=1, cap=budget + 2)
    st = cd.alloc_layer_state(p)
    ws = torch.empty((cd.calidrop_accumulated_scores_workspace_bytes(p),), dtype=torch.uint8, device="cuda")
    scores = torch.full((B, Hkv, L), -1.0, dtype=torch.float32, device="cuda")
    runs = []
    for _ in range(2):                                  # twice: the result is reproducible bit for bit
        cd.calidrop_accumulated_scores(p, to_dev(Qf), to_dev(Kb), scores, ws)
        torch.cuda.synchronize()
        runs.append(scores.cpu().numpy().copy())
    np.testing.assert_array_equal(runs[0], runs[1])
    got = runs[0]
    ref = np.stack([np.stack([oracle.accumulated_attention(Qf[b, h * G:(h + 1) * G], Kb[b, h]) for h in range(Hkv)])
                    for b in range(B)])
    # every query's attention sums to one: the scores of a kv head sum to G * L
    np.testing.assert_allclose(ref.sum(-1), G * L, rtol=1e-9)
    np.testing.assert_allclose(got, ref, rtol=2e-5, atol=1e-6)
    np.testing.assert_allclose(got.sum(-1, dtype=np.float64), G * L, rtol=1e-5)
    cd.calidrop_select_from_scores(p, scores, budget // 2, st.kept_idx, st.ws_compress)
    torch.cuda.synchronize()
    kept = st.kept_idx.cpu().numpy()
    for b in range(B):
        for h in range(Hkv):
            want = oracle.select_from_scores(ref[b, h].astype(np.float32), tail=budget // 2, budget=budget)
            a, w = set(kept[b, h].tolist()), set(want.tolist())
            assert len(a) == budget and np.all(np.diff(kept[b, h]) > 0)
            if a != w:                                  # only near-ties of the oracle's scores may swap
                thr = min(ref[b, h][t] for t in w if t < L - budget // 2)
                for t in a ^ w:
                    assert abs(ref[b, h][t] - thr) <= 2e-5 * thr, (b, h, t, ref[b, h][t], thr)
    # argument checks
    small = torch.empty((16,), dtype=torch.uint8, device="cuda")
    assert cd.calidrop_accumulated_scores(p, to_dev(Qf), to_dev(Kb), scores, small, check=False) == cd.WORKSPACE_TOO_SMALL
    assert cd.calidrop_accumulated_scores(p, None, to_dev(Kb), scores, ws, check=False) == cd.INVALID_ARG


@pytest.mark.parametrize("B,Hq,Hkv,L", [
    (1, 1, 1, 1),        # a single key
    (1, 2, 1, 127),      # one partial row tile
    (1, 3, 3, 128),      # full row tile, half a column tile
    (2, 2, 1, 129),      # the second row tile holds one row, its job's second half is not seen
    (1, 2, 2, 257),      # the second column tile holds one column
    (2, 40, 8, 1025),    # 720 items: several per CTA, forwards and backwards, with odd and even job counts
])
def test_accumulated_scores_at_the_edges_of_their_tiles(cuda_lib, B, Hq, Hkv, L):
    """Against attention in fp64.  A score sums up to G L probabilities, each with a relative error of about 2^-22
    from exp2, 2^-24 |logit| from the fp32 logits and statistics; 2e-5 covers them tenfold."""
    cd = cuda_lib
    gen = torch.Generator(device="cuda").manual_seed(L)
    Q = (2.0 * torch.randn((B, Hq, L, 128), generator=gen, device="cuda")).to(torch.bfloat16)
    K = torch.randn((B, Hkv, L, 128), generator=gen, device="cuda").to(torch.bfloat16)
    p = cd.make_params(B=B, Hq=Hq, Hkv=Hkv, L=L, window=1, pool=1, budget=L, n_cal=1, cap=L)
    ws = torch.empty((cd.calidrop_accumulated_scores_workspace_bytes(p),), dtype=torch.uint8, device="cuda")
    scores = torch.full((B, Hkv, L), -1.0, dtype=torch.float32, device="cuda")
    cd.calidrop_accumulated_scores(p, Q, K, scores, ws)
    G = Hq // Hkv
    ref = torch.zeros((B, Hkv, L), dtype=torch.float64, device="cuda")
    mask = torch.ones((L, L), dtype=torch.bool, device="cuda").triu(1)
    for b in range(B):
        for hq in range(Hq):
            s = (Q[b, hq].double() @ K[b, hq // G].double().T) / 128 ** 0.5
            ref[b, hq // G] += torch.softmax(s.masked_fill_(mask, -float("inf")), -1).sum(0)
    torch.testing.assert_close(scores.double(), ref, rtol=2e-5, atol=1e-6)


def test_a_thread_may_start_with_a_call_of_the_library(cuda_lib):
    """A thread that has made no other CUDA call has no current context yet; prompts and decode steps alike."""
    cd = cuda_lib
    cfg = wl.small_config()
    Q, K, V = _inputs(cfg)
    args = dict(window=8, pool=5, budget=40, n_cal=1, cap=42)
    want = gpu_compress(Q, K, V, **args)
    st, p = want.st, want.p
    dQ, dK, dV = to_dev(Q), to_dev(K), to_dev(V)
    q = dQ[:, :, -1].contiguous()
    out = torch.empty((2,) + tuple(q.shape), dtype=torch.bfloat16, device="cuda")
    K_kept, V_kept = st.K_kept.clone(), st.V_kept.clone()      # caches whose descriptors no call has made yet
    st2 = cd.alloc_layer_state(p)
    torch.cuda.synchronize()
    errors = []

    def work(f):
        try:
            f()
        except Exception as e:
            errors.append(e)

    def decode(kc, vc, o):
        cd.calidrop_decode(p, q, None, None, kc, vc, 40, st.O_c, st.LSE_c, st.C_q, o, None, None, st.ws_decode)

    for f in (lambda: cd.calidrop_compress(p, dQ, dK, dV, None, st2.kept_idx, st2.K_kept, st2.V_kept, st2.O_c, st2.LSE_c, st2.C_q,
                                           st2.ws_compress),
              lambda: decode(K_kept, V_kept, out[0])):
        t = threading.Thread(target=work, args=(f,))
        t.start()
        t.join()
    assert not errors, errors
    decode(st.K_kept, st.V_kept, out[1])
    assert torch.equal(st2.kept_idx, st.kept_idx) and torch.equal(st2.O_c, st.O_c) and torch.equal(out[0], out[1])


def test_first_calls_of_several_threads_with_different_window_sizes(cuda_lib):
    """Threads whose first calls need different amounts of shared memory of the same kernel start at the same moment, in a
    process of its own (what a launch sets up once per device is not set up yet there).  (The two can interleave in
    an order that leaves the lower limit; whether they do is up to the scheduler.)"""
    code = """
import threading, torch
from paper_2507_19906_b200 import binding as cd
cd.load()
L, W, budget, out, errors = 700, 32, 80, {}, []
def state(G):
    gen = torch.Generator(device="cuda").manual_seed(G)
    rn = lambda *sh: torch.randn(sh, generator=gen, device="cuda").to(torch.bfloat16)
    p = cd.make_params(B=1, Hq=G, Hkv=1, L=L, window=W, pool=1, budget=budget, n_cal=W, cap=budget)
    return p, rn(1, G, W, 128), rn(1, 1, L, 128), rn(1, 1, L, 128), cd.alloc_layer_state(p)
def run(p, Q, K, V, st):
    cd.calidrop_compress(p, Q, K, V, None, st.kept_idx, st.K_kept, st.V_kept, st.O_c, st.LSE_c, st.C_q, st.ws_compress)
states = {G: state(G) for G in range(1, 9)}
torch.cuda.synchronize()
start = threading.Barrier(len(states))
def work(G):
    with torch.cuda.stream(torch.cuda.Stream()):
        torch.zeros(1, device="cuda")
        start.wait()
        try:
            for _ in range(20): run(*states[G])
        except Exception as e:
            errors.append((G, e))
threads = [threading.Thread(target=work, args=(G,)) for G in states]
[t.start() for t in threads]; [t.join() for t in threads]
torch.cuda.synchronize()
assert not errors, errors
for G, s in states.items():
    got = [t.clone() for t in (s[4].kept_idx, s[4].O_c, s[4].LSE_c)]
    run(*s)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(got, (s[4].kept_idx, s[4].O_c, s[4].LSE_c))), G
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    subprocess.run([sys.executable, "-c", code], cwd=root, check=True, timeout=300)


@pytest.mark.parametrize("Hq,one_kernel", [(8, True), (10, False)])
def test_calls_enqueued_back_to_back_give_the_results_of_calls_run_one_at_a_time(cuda_lib, Hq, one_kernel):
    """The kernels of a compress call start beside the end of their predecessors (programmatic dependent
    launch) and a decode launch prefetches ahead of its dependency wait: a stream of calls with no
    synchronisation between them, on one shared workspace, must leave exactly what the same calls leave
    when each is waited for."""
    cd = cuda_lib
    B, Hkv, L, W, pool, budget, n_cal = 2, 2, 2300, 32, 7, 256, 32
    cfgs = [wl.small_config(B=B, Hq=Hq, Hkv=Hkv, L=L, window=W, pool=pool, budget=budget, steps=3, n_heavy=24,
                            seed=s) for s in (5, 6)]
    inputs = [tuple(to_dev(x) for x in _inputs(c)) for c in cfgs]
    T = 3
    p = cd.make_params(B=B, Hq=Hq, Hkv=Hkv, L=L, window=W, pool=pool, budget=budget, n_cal=n_cal, cap=budget + T)
    dec = [tuple(to_dev(x) for x in wl.gen_decode_inputs(c, wl.gen_q_obs(c), steps=T)) for c in cfgs]

    def run(sync):
        states = [cd.alloc_layer_state(p) for _ in range(2)]
        for st in states:
            st.ws_compress = states[0].ws_compress          # one workspace for every call
        outs = []
        for rnd in range(3):
            for i, (st, (dQ, dK, dV)) in enumerate(zip(states, inputs)):
                before = cd.calidrop_launch_count()
                cd.calidrop_compress(p, dQ, dK, dV, None, st.kept_idx, st.K_kept, st.V_kept, st.O_c, st.LSE_c, st.C_q,
                                     st.ws_compress)
                assert (cd.calidrop_launch_count() - before == 1) == one_kernel
                if sync:
                    torch.cuda.synchronize()
                q, kn, vn = dec[i]
                for t in range(T):
                    o = torch.empty((B, Hq, 128), dtype=torch.bfloat16, device="cuda")
                    cd.calidrop_decode(p, q[t], kn[t], vn[t], st.K_kept, st.V_kept, budget + t, st.O_c, st.LSE_c,
                                       st.C_q, o, None, None, st.ws_decode)
                    if sync:
                        torch.cuda.synchronize()
                    outs.append(o)
        torch.cuda.synchronize()
        lay = cd.calidrop_compress_workspace_layout(p)
        assert int(states[0].ws_compress[lay.status_offset: lay.status_offset + 4].view(torch.int32).item()) == 0
        return states, outs

    ref_states, ref_outs = run(sync=True)
    got_states, got_outs = run(sync=False)
    for a, b in zip(ref_states, got_states):
        assert torch.equal(a.kept_idx, b.kept_idx)
        assert torch.equal(a.K_kept, b.K_kept) and torch.equal(a.V_kept, b.V_kept)
        assert torch.equal(a.O_c, b.O_c) and torch.equal(a.LSE_c, b.LSE_c) and torch.equal(a.C_q, b.C_q)
    for a, b in zip(ref_outs, got_outs):
        assert torch.equal(a, b)


# ---------------------------------------------------------------- seeded random shapes
def _random_shapes(n, seed):
    rng = np.random.Generator(np.random.Philox(key=[seed, 1]))
    out = []
    for _ in range(n):
        Hkv = int(rng.integers(1, 5))
        G = int(rng.integers(1, 9))
        B = int(rng.integers(1, 4))
        W = int(rng.choice([1, 2, 4, 8, 16, 32, 64]))
        if G * W > 512:
            W = 512 // G
        L = int(rng.integers(W + 40, 2600))
        budget = int(rng.integers(W + 1, min(L, W + 700)))
        pool = int(rng.choice([1, 3, 5, 7]))
        n_cal = int(rng.integers(1, W + 1))
        out.append((B, Hkv * G, Hkv, L, W, pool, budget, n_cal))
    return out


@pytest.mark.parametrize("B,Hq,Hkv,L,W,pool,budget,n_cal", _random_shapes(16, 2507))
def test_compress_and_decode_random_shapes(cuda_lib, B, Hq, Hkv, L, W, pool, budget, n_cal):
    cfg = wl.small_config(B=B, Hq=Hq, Hkv=Hkv, L=L, window=W, pool=pool, budget=budget, steps=3,
                          n_sink=2, n_heavy=max(1, L // 50))
    Q, K, V = _inputs(cfg)
    T = 3
    g = gpu_compress(Q, K, V, window=W, pool=pool, budget=budget, n_cal=n_cal, cap=budget + T)
    ref, _ = compare_compress(g, Q, K, V, window=W, pool=pool, budget=budget, n_cal=n_cal)
    q, kn, vn = wl.gen_decode_inputs(cfg, Q, steps=T)
    st = decode_steps_compare(g, ref, q, kn, vn, steps=T)
    assert st["total"] == T * B * Hq
