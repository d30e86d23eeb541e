"""The work that users have this library do, as cases whose time can be measured.

Every case is one pass through the public entry points of `paper_2507_19906_b200.binding`:

  compress    the end-of-prefill step of one attention layer (calidrop_compress)
  decode      one token through `layers` attention layers, one calidrop_decode call per layer, or
              (`batched`) one calidrop_decode_batched launch for all of them
  recompute   the evicted rows compacted for the offload, one calibration entry recomputed from
              them, and the decode step repeated (calidrop_gather_evicted, calidrop_recalibrate,
              calidrop_decode)
  h2o         the accumulated-attention eviction rule: scores of a whole prompt, kept list, gather and
              calibration (calidrop_accumulated_scores, calidrop_select_from_scores, calidrop_calibrate)

The inputs follow the statistics of `workload.py`: a base direction per query head that nearby queries
share, unit-normal keys and values, attention sinks, and heavy hitters that carry about half of the
attention mass.  There are half as many heavy hitters again as a budget holds and their weights are
spread over a factor of ten, so the boundary of the kept set lies among them.
"""
from __future__ import annotations

import math

import torch

from paper_2507_19906_b200 import binding as cd

D = 128

_COMPRESS = dict(kind="compress", pool=7, n_cal=1, lse=False, calib_size=0)
_DECODE = dict(kind="decode", layers=1, batched=False, append=True)


def listed():
    return [
        # short prompt, every head its own keys, the last query alone calibrates: launches and latency
        dict(_COMPRESS, name="compress 2k", B=1, Hq=8, Hkv=8, L=2048, window=32, budget=128),
        # one request of an ordinary prompt
        dict(_COMPRESS, name="compress 8k", B=1, Hq=32, Hkv=8, L=8192, window=32, budget=512, n_cal=32),
        # ragged sizes and the options: row LSE handed over by the prefill, calibration size of Section 4.4
        dict(_COMPRESS, name="compress ragged", B=2, Hq=40, Hkv=8, L=5003, window=24, pool=5, budget=300, n_cal=8,
             lse=True, calib_size=1000),
        # a batch whose prefill hands over its row LSE, small budget
        dict(_COMPRESS, name="compress 16k b8", B=8, Hq=32, Hkv=8, L=16384, window=32, budget=128, n_cal=32, lse=True),
        # a batch of long prompts, every window query calibrates
        dict(_COMPRESS, name="compress 32k b4", B=4, Hq=32, Hkv=8, L=32768, window=64, budget=2048, n_cal=64),
        # one very long prompt, seven query heads per kv head
        dict(_COMPRESS, name="compress 131k", B=1, Hq=28, Hkv=4, L=131072, window=64, budget=4096, n_cal=64),
        # the smallest decode call
        dict(_DECODE, name="decode 128", B=1, Hq=8, Hkv=8, kv=128, n_cal=1),
        # one token of a batch through eight layers, called layer by layer
        dict(_DECODE, name="decode 2k b4", B=4, Hq=32, Hkv=8, kv=2111, n_cal=64, layers=8),
        # few kv heads with a long retained cache
        dict(_DECODE, name="decode 4k", B=1, Hq=28, Hkv=4, kv=4333, n_cal=64, layers=8),
        # a whole stack of small caches in one launch
        dict(_DECODE, name="decode stack", B=8, Hq=32, Hkv=8, kv=231, n_cal=32, layers=32, batched=True),
        # the query drifted: offload compaction, recompute, decode again
        dict(kind="recompute", name="recompute 32k b4", B=4, Hq=32, Hkv=8, L=32768, window=64, budget=2048, n_cal=64),
        # another eviction rule, from the queries of the whole prompt
        dict(kind="h2o", name="h2o 8k", B=1, Hq=32, Hkv=8, L=8192, window=32, budget=512, n_cal=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["compress"] * 6 + ["decode"] * 4 + ["recompute", "h2o"])
    Hq, Hkv = rng.choice([(8, 8), (32, 8), (40, 8), (28, 4), (16, 2), (24, 8), (12, 4), (32, 32)])
    window = rng.choice([8, 16, 24, 32, 32, 64])
    n_cal = rng.choice([1, window, rng.randint(1, window)])
    if kind == "decode":
        batched = rng.random() < 0.4
        B = rng.choice([1, 1, 2, 3, 4, 8])
        layers = _log(rng, 2, 32) if batched else _log(rng, 1, 12)
        rows = 32 * 64 * 231                      # rows over all units and layers of the largest listed case
        kv = _log(rng, 100, max(128, min(16000, rows // (B * Hkv * layers))))
        return dict(_DECODE, B=B, Hq=Hq, Hkv=Hkv, kv=kv, n_cal=n_cal, layers=layers, batched=batched,
                    append=rng.random() < 0.8)
    if kind == "h2o":
        L = _log(rng, 600, 8192)
        B = rng.choice([1, 1, 2])
        while B * Hq * L * L > 32 * 8192 * 8192:
            L = L * 2 // 3
        return dict(kind="h2o", B=B, Hq=Hq, Hkv=Hkv, L=L, window=window, budget=_log(rng, 2 * window + 32, L // 3),
                    n_cal=n_cal)
    B = rng.choice([1, 1, 2, 4, 8])
    L = _log(rng, 1024, 131072)
    while B * Hkv * L > 32 * 32768 or B * Hq * window * L > 128 * 64 * 32768:
        L = L * 2 // 3
    budget = _log(rng, window + 64, max(window + 128, min(4096, L // 4)))
    if kind == "recompute":
        return dict(kind="recompute", B=B, Hq=Hq, Hkv=Hkv, L=L, window=window, budget=budget, n_cal=n_cal)
    return dict(_COMPRESS, B=B, Hq=Hq, Hkv=Hkv, L=L, window=window, pool=rng.choice([1, 3, 5, 7, 7]), budget=budget,
                n_cal=n_cal, lse=rng.random() < 0.35, calib_size=rng.choice([0, 0, 0, _log(rng, 64, max(65, L // 3))]))


# ------------------------------------------------------------------------------------ inputs
class _Gen:
    """Seeded normal numbers on the GPU."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda").manual_seed(seed)

    def normal(self, *shape):
        return torch.randn(shape, generator=self.g, device="cuda")

    def perm(self, n):
        return torch.randperm(n, generator=self.g, device="cuda")


def _prompt(gen, c, u, n_sel):
    """K and V [B, Hkv, L, D] of a prompt whose queries look along u [B, Hq, D]: unit-normal rows, eight
    sinks, and heavy hitters enough for 1.5 times the `n_sel` rows a selection takes (each of them lifts
    the `pool` rows around it)."""
    B, Hkv, L = c["B"], c["Hkv"], c["L"]
    K = torch.empty((B, Hkv, L, D), dtype=torch.bfloat16, device="cuda")
    V = torch.empty_like(K)
    n_cand = L - c["window"]
    n_heavy = min(n_cand // 2, int(1.5 * n_sel / c.get("pool", 1)) + 16)
    dirs = u.view(B, Hkv, -1, D).sum(2)                          # the direction a kv head's queries share
    # softmax weight of a heavy hitter: about n_cand / n_heavy times a bulk row's, a factor e of spread;
    # a key of `a` times the shared direction has the logit a * |u|^2 / sqrt(D) = a * sqrt(D)
    level = (0.54 + math.log(n_cand / n_heavy)) / math.sqrt(D)
    for b in range(B):
        K[b] = gen.normal(Hkv, L, D)
        V[b] = gen.normal(Hkv, L, D)
        for h in range(Hkv):
            pos = gen.perm(n_cand)[:n_heavy]
            amp = level + gen.normal(n_heavy, 1) / math.sqrt(D)
            K[b, h, pos] = (amp * dirs[b, h] + 0.3 * gen.normal(n_heavy, D)).to(torch.bfloat16)
            K[b, h, :8] = (0.5 * dirs[b, h]).to(torch.bfloat16)
    return K, V


def _row_lse(Q, K, window):
    """What a prefill attention hands over: natural-log softmax denominators of the window rows."""
    B, Hq, W, _ = Q.shape
    Hkv, L = K.shape[1], K.shape[2]
    out = torch.empty((B, Hq, W), dtype=torch.float32, device="cuda")
    seen = torch.arange(L, device="cuda")[None, :] <= L - W + torch.arange(W, device="cuda")[:, None]
    for b in range(B):
        for hq in range(Hq):
            s = (Q[b, hq].float() @ K[b, hq // (Hq // Hkv)].float().T) / math.sqrt(D)
            out[b, hq] = torch.logsumexp(s.masked_fill_(~seen, -math.inf), -1)
    return out


def _calibration(gen, lead, n_cal):
    """A calibration state as compress leaves it: nearby queries share a direction, and so their outputs
    and normalisers are close.  Returns C_q, O_c, LSE_c and the direction."""
    u = gen.normal(*lead, D)
    C_q = (u[..., None, :] + 0.3 * gen.normal(*lead, n_cal, D)).to(torch.bfloat16)
    O_c = 0.1 * gen.normal(*lead, 1, D) + 0.01 * gen.normal(*lead, n_cal, D)
    LSE_c = 9.0 + 0.3 * gen.normal(*lead, 1) + 0.05 * gen.normal(*lead, n_cal)
    return C_q, O_c.contiguous(), LSE_c.contiguous(), u


def _prepare_compress(c, seed):
    gen = _Gen(seed)
    u = gen.normal(c["B"], c["Hq"], D)
    K, V = _prompt(gen, c, u, c["budget"] - c["window"])
    Q = (u[:, :, None, :] + 0.3 * gen.normal(c["B"], c["Hq"], c["window"], D)).to(torch.bfloat16)
    p = cd.make_params(B=c["B"], Hq=c["Hq"], Hkv=c["Hkv"], L=c["L"], window=c["window"], pool=c["pool"],
                       budget=c["budget"], n_cal=c["n_cal"], cap=c["budget"], calib_size=c["calib_size"])
    return dict(c=c, p=p, Q=Q, K=K, V=V, lse=_row_lse(Q, K, c["window"]) if c["lse"] else None,
                st=cd.alloc_layer_state(p))


def _run_compress(s):
    st = s["st"]
    cd.calidrop_compress(s["p"], s["Q"], s["K"], s["V"], s["lse"], st.kept_idx, st.K_kept, st.V_kept, st.O_c, st.LSE_c,
                         st.C_q, st.ws_compress)
    return st.kept_idx, st.K_kept, st.V_kept, st.O_c, st.LSE_c, st.C_q


def _prepare_decode(c, seed):
    gen = _Gen(seed)
    n, B, Hq, Hkv, cap = c["layers"], c["B"], c["Hq"], c["Hkv"], c["kv"] + 8
    K, V = (torch.zeros((n, B, Hkv, cap, D), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    for i in range(n):
        K[i, :, :, :c["kv"]] = gen.normal(B, Hkv, c["kv"], D)
        V[i, :, :, :c["kv"]] = gen.normal(B, Hkv, c["kv"], D)
    C_q, O_c, LSE_c, u = _calibration(gen, (n, B, Hq), c["n_cal"])
    q = (u + 0.3 * gen.normal(n, B, Hq, D)).to(torch.bfloat16)
    kn, vn = (gen.normal(n, B, Hkv, D).to(torch.bfloat16) for _ in range(2))
    p = cd.make_params(B=B, Hq=Hq, Hkv=Hkv, n_cal=c["n_cal"], cap=cap)
    out = torch.empty((n, B, Hq, D), dtype=torch.bfloat16, device="cuda")
    lse = torch.empty((n, B, Hq), dtype=torch.float32, device="cuda")
    flags = torch.empty((n, B, Hq), dtype=torch.uint8, device="cuda")
    ws = torch.zeros((cd.calidrop_decode_workspace_bytes(p, cap) * (n if c["batched"] else 1),), dtype=torch.uint8,
                     device="cuda")
    layers = [dict(q=q[i], k_new=kn[i] if c["append"] else None, v_new=vn[i] if c["append"] else None, K_kept=K[i],
                   V_kept=V[i], O_c=O_c[i], LSE_c=LSE_c[i], C_q=C_q[i], out=out[i], lse_out=lse[i], flags=flags[i])
              for i in range(n)]
    return dict(c=c, p=p, layers=layers, array=cd.make_decode_layers(layers), ws=ws, K=K, V=V, out=out, lse=lse,
                flags=flags, keep=(q, kn, vn, C_q, O_c, LSE_c))


def _run_decode(s):
    c = s["c"]
    if c["batched"]:
        cd.calidrop_decode_batched(s["p"], s["array"], c["kv"], s["ws"])
    else:
        for d in s["layers"]:
            cd.calidrop_decode(s["p"], d["q"], d["k_new"], d["v_new"], d["K_kept"], d["V_kept"], c["kv"], d["O_c"],
                               d["LSE_c"], d["C_q"], d["out"], d["lse_out"], d["flags"], s["ws"])
    return s["out"], s["lse"], s["flags"], s["K"], s["V"]


def _prepare_recompute(c, seed):
    gen = _Gen(seed)
    B, Hq, Hkv, L, W, budget = (c[k] for k in ("B", "Hq", "Hkv", "L", "window", "budget"))
    C_q, O_c, LSE_c, u = _calibration(gen, (B, Hq), c["n_cal"])
    K, V = _prompt(gen, c, u, budget - W)
    kept = torch.empty((B, Hkv, budget), dtype=torch.int32, device="cuda")
    kept[:, :, budget - W:] = torch.arange(L - W, L, device="cuda")
    for b in range(B):
        for h in range(Hkv):
            kept[b, h, :budget - W] = gen.perm(L - W)[:budget - W].sort().values
    p = cd.make_params(B=B, Hq=Hq, Hkv=Hkv, L=L, window=W, pool=7, budget=budget, n_cal=c["n_cal"], cap=budget + 8)
    st = cd.alloc_layer_state(p)
    st.kept_idx.copy_(kept)
    st.C_q.copy_(C_q), st.O_c.copy_(O_c), st.LSE_c.copy_(LSE_c)
    rows = kept.long()[..., None].expand(-1, -1, -1, D)
    st.K_kept[:, :, :budget] = K.gather(2, rows)
    st.V_kept[:, :, :budget] = V.gather(2, rows)
    bf = dict(dtype=torch.bfloat16, device="cuda")
    return dict(c=c, p=p, K=K, V=V, st=st, n_evict=L - budget,
                q=(0.5 * u + gen.normal(B, Hq, D)).to(torch.bfloat16),
                kn=gen.normal(B, Hkv, D).to(torch.bfloat16), vn=gen.normal(B, Hkv, D).to(torch.bfloat16),
                evict_idx=torch.empty((B, Hkv, L - budget), dtype=torch.int32, device="cuda"),
                K_evict=torch.empty((B, Hkv, L - budget, D), **bf), V_evict=torch.empty((B, Hkv, L - budget, D), **bf),
                out=torch.empty((B, Hq, D), **bf), lse=torch.empty((B, Hq), dtype=torch.float32, device="cuda"),
                flags=torch.empty((B, Hq), dtype=torch.uint8, device="cuda"))


def _run_recompute(s):
    p, st, c = s["p"], s["st"], s["c"]
    cd.calidrop_gather_evicted(p, s["K"], s["V"], st.kept_idx, s["evict_idx"], s["K_evict"], s["V_evict"],
                               st.ws_compress)
    cd.calidrop_recalibrate(p, s["q"], s["K_evict"], s["V_evict"], s["n_evict"], c["n_cal"] - 1, st.O_c, st.LSE_c,
                            st.C_q, st.ws_decode)
    cd.calidrop_decode(p, s["q"], s["kn"], s["vn"], st.K_kept, st.V_kept, c["budget"], st.O_c, st.LSE_c, st.C_q,
                       s["out"], s["lse"], s["flags"], st.ws_decode)
    return (s["evict_idx"], s["K_evict"], s["V_evict"], st.O_c, st.LSE_c, st.C_q, s["out"], s["lse"], s["flags"],
            st.K_kept, st.V_kept)


def _prepare_h2o(c, seed):
    gen = _Gen(seed)
    B, Hq, Hkv, L, W, budget = (c[k] for k in ("B", "Hq", "Hkv", "L", "window", "budget"))
    u = gen.normal(B, Hq, D)
    K, V = _prompt(gen, c, u, budget - max(W, budget // 2))
    Q = torch.empty((B, Hq, L, D), dtype=torch.bfloat16, device="cuda")
    for b in range(B):
        Q[b] = u[b][:, None, :] + 0.3 * gen.normal(Hq, L, D)
    p = cd.make_params(B=B, Hq=Hq, Hkv=Hkv, L=L, window=W, pool=1, budget=budget, n_cal=c["n_cal"], cap=budget)
    return dict(c=c, p=p, Q=Q, Q_obs=Q[:, :, L - W:].contiguous(), K=K, V=V, st=cd.alloc_layer_state(p),
                scores=torch.empty((B, Hkv, L), dtype=torch.float32, device="cuda"),
                ws=torch.empty((cd.calidrop_accumulated_scores_workspace_bytes(p),), dtype=torch.uint8, device="cuda"))


def _run_h2o(s):
    p, st, c = s["p"], s["st"], s["c"]
    cd.calidrop_accumulated_scores(p, s["Q"], s["K"], s["scores"], s["ws"])
    cd.calidrop_select_from_scores(p, s["scores"], max(c["window"], c["budget"] // 2), st.kept_idx, st.ws_compress)
    cd.calidrop_calibrate(p, s["Q_obs"], s["K"], s["V"], None, st.kept_idx, st.K_kept, st.V_kept, st.O_c, st.LSE_c,
                          st.C_q, st.ws_compress)
    return s["scores"], st.kept_idx, st.K_kept, st.V_kept, st.O_c, st.LSE_c, st.C_q


_KINDS = {
    "compress": (_prepare_compress, _run_compress),
    "decode": (_prepare_decode, _run_decode),
    "recompute": (_prepare_recompute, _run_recompute),
    "h2o": (_prepare_h2o, _run_h2o),
}


def prepare(case, seed):
    state = _KINDS[case["kind"]][0](case, seed)
    state["run"] = _KINDS[case["kind"]][1]
    return state


def run(state):
    return state["run"](state)


# ------------------------------------------------------------------------------------ work and tolerance
def _compress_work(c, E):
    """Window scoring, pooled top-k, gather, calibration over E rows per kv head."""
    units, rows = c["B"] * c["Hkv"], c["B"] * c["Hq"]
    flops = 2 * rows * c["window"] * c["L"] * D + 2 * rows * c["n_cal"] * E * D
    byts = (2 * rows * c["window"] * D + 2 * units * (c["L"] + E + c["budget"]) * D      # queries, K, the V rows used
            + 4 * units * c["budget"] * (D + 1) + rows * c["n_cal"] * (4 * D + 4 + 2 * D))
    return byts + (4 * rows * c["window"] if c.get("lse") else 0), flops


def _decode_work(c, kv):
    units, rows = c["B"] * c["Hkv"], c["B"] * c["Hq"]
    return 4 * units * kv * D + rows * (2 * D + 2 * c["n_cal"] * D + 4 * D + 4 + 2 * D + 5), 4 * rows * kv * D


def work(case):
    c = case
    if c["kind"] == "compress":
        E = c["L"] - c["budget"]
        b, f = _compress_work(c, min(c["calib_size"], E) if c["calib_size"] else E)
    elif c["kind"] == "decode":
        b, f = _decode_work(c, c["kv"] + (1 if c["append"] else 0))
        b, f = b * c["layers"], f * c["layers"]
    elif c["kind"] == "recompute":
        n_e, units, rows = c["L"] - c["budget"], c["B"] * c["Hkv"], c["B"] * c["Hq"]
        b, f = _decode_work(c, c["budget"] + 1)
        # the evicted rows read and written, their indices written
        b += 2 * 4 * units * n_e * D + 4 * units * (n_e + c["budget"]) + rows * (8 * D + 4)
        f += 4 * rows * n_e * D
    else:
        # causal logits of every prompt query once, then the calibration step (its logits are among them)
        rows = c["B"] * c["Hq"]
        b, _ = _compress_work(c, c["L"] - c["budget"])
        b += 2 * rows * c["L"] * D + 4 * c["B"] * c["Hkv"] * c["L"]
        f = rows * c["L"] * c["L"] * D + 2 * rows * c["n_cal"] * (c["L"] - c["budget"]) * D
    return {"bytes": b, "flops": f}


def tolerance(case):
    """bf16 probabilities in the value products and bf16 outputs; kept rows, indices and flags may differ
    where two candidates tie to the last bits of the fp32 scores."""
    return {"rel": 6e-3, "max": 0.2, "differ": 2e-3}
