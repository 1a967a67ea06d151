"""The work that a user of this library has it do, as cases that can be timed and compared.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges.  A case is one call (or
the few calls that belong together) of the public entry points in ``paper_2601_21896_b200.binding``,
on device buffers that the program keeps between calls.  Sizes are the repository's own
configurations (``workloads.py``: 1560 tokens a frame, chunks of 4680, 12 heads x 128 or 40 x 128)
and ragged small ones; per-stream sizes are texts of comma-separated numbers.
"""
import math

import numpy as np
import torch

from paper_2601_21896_b200 import binding as B
from paper_2601_21896_b200 import workloads as wl
from paper_2601_21896_b200.harness import Layer

PAPER_HIDDEN, PAPER_OUT = 1024, 12      # the paper's head: [q, k, v] -> 1024 -> 12, SiLU


def listed():
    return [
        # the smallest call: one layer of the Tiny configuration, d_head 64, sigmoid scores; latency only
        dict(name="tiny_step", op="step", heads=2, d_head=64, T="512", budget="128", sink=4, recent=64, Lq="64",
             hidden=32, sigmoid=True, frame=64, structure="iid", q_gain=1.0, lse=False),
        # three ragged streams with odd lengths (one of them not pruned): a small batch of short videos
        dict(name="ragged_step", op="step", heads=2, d_head=128, T="700,333,1200", budget="300,333,517", sink=24,
             recent=72, Lq="200,72,331", hidden=64, sigmoid=False, frame=24, structure="lowrank", q_gain=2.0, lse=True),
        # one layer of one denoising step at the paper's cache size: attention only (pruning happens
        # once a chunk), peaked rows
        dict(name="denoise_attn", op="attn", heads=12, d_head=128, B="4680", Lq="4680", q_gain=2.0, lse=False),
        # one layer step at the paper's own operating point, 9360 -> 4680, no recent window
        dict(name="paper_step", op="step", heads=12, d_head=128, T="9360", budget="4680", sink=1560, recent=0,
             Lq="4680", hidden=256, sigmoid=False, frame=1560, structure="lowrank", q_gain=1.0, lse=False),
        # the headline: one Wan-1.3B-class layer, 28080 -> 14040
        dict(name="wan_step", op="step", heads=12, d_head=128, T="28080", budget="14040", sink=1560, recent=4680,
             Lq="4680", hidden=256, sigmoid=False, frame=1560, structure="lowrank", q_gain=1.0, lse=False),
        # the same cache at a quarter of the tokens, attention through the index list (no second copy
        # of the cache)
        dict(name="wan_step_indexed", op="step_indexed", heads=12, d_head=128, T="28080", budget="7020", sink=1560,
             recent=4680, Lq="4680", hidden=256, sigmoid=False, frame=1560, structure="lowrank", q_gain=1.0, lse=False),
        # a long video: 60 frames of cache pruned to 6
        dict(name="long_horizon_step", op="step", heads=12, d_head=128, T="93600", budget="9360", sink=1560,
             recent=4680, Lq="4680", hidden=256, sigmoid=False, frame=1560, structure="lowrank_ar1", q_gain=1.0, lse=False),
        # the largest: four ragged streams of a 14B-class layer
        dict(name="batch4_step", op="step", heads=40, d_head=128, T="9360,18720,28080,46800",
             budget="3276,6552,9828,16380", sink=1560, recent=1560, Lq="4680,4680,4680,4680", hidden=512, sigmoid=False,
             frame=1560, structure="lowrank", q_gain=1.0, lse=False),
        # once per generated chunk: score the chunk with the paper's head, prune all 30 layers' caches
        # with one index list, append the chunk's rows
        dict(name="cache_update", op="cache_update", layers=30, heads=12, d_head=128, capacity=9360, chunk=4680, sink=1560),
        # training: the teacher's salience target over 9 frames, row statistics computed by the call
        dict(name="teacher_salience", op="sse", heads=12, L=14040, block=4680, with_lse=False, pools=False),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _csv(values):
    return ",".join(str(int(v)) for v in values)


def _ints(text):
    return tuple(int(v) for v in text.split(","))


def draw(rng):
    """One more case of the listed ranges; never more work than the largest listed one."""
    most = max(work(c)["flops"] for c in listed())
    while True:
        c = _draw_any(rng)
        w = work(c)
        if w["flops"] <= 0.9 * most and w["bytes"] <= 8e9:
            return c


def _draw_any(rng):
    op = rng.choice(["step", "step", "step", "step_indexed", "attn", "attn", "cache_update", "sse"])
    gain = rng.choice([1.0, 1.0, 2.0, 4.0])
    if op == "cache_update":
        chunk = _logint(rng, 64, 4680)
        capacity = chunk + _logint(rng, 64, 14040)
        return dict(op=op, layers=rng.randint(1, 30), heads=rng.choice([2, 6, 12, 16]), d_head=128, capacity=capacity,
                    chunk=chunk, sink=min(1560, (capacity - chunk) // 3))
    if op == "sse":
        L = _logint(rng, 700, 14040)
        return dict(op=op, heads=rng.choice([2, 5, 12]), L=L, block=min(L, _logint(rng, 200, 4680)),
                    with_lse=rng.random() < 0.5, pools=rng.random() < 0.25)
    d_head = 64 if op != "step_indexed" and rng.random() < 0.2 else 128
    heads = rng.choice([2, 4, 12]) if d_head == 64 else rng.choice([2, 5, 12, 24, 40])
    n = rng.choice([1, 1, 1, 2, 4])
    lq = _csv(_logint(rng, 64, 4680) for _ in range(n))
    if op == "attn":
        return dict(op=op, heads=heads, d_head=d_head, B=_csv(_logint(rng, 128, 28080) for _ in range(n)), Lq=lq,
                    q_gain=gain, lse=rng.random() < 0.5)
    T = [_logint(rng, 512, 93600) for _ in range(n)]
    budget = [max(64, int(t * rng.uniform(0.1, 0.75))) for t in T]
    least = min(budget)
    recent = rng.choice([0, least // 5, least // 3])
    return dict(op=op, heads=heads, d_head=d_head, T=_csv(T), budget=_csv(budget), sink=min(1560, least // 6), recent=recent,
                Lq=lq, hidden=rng.choice([32, 64, 256, 512]), sigmoid=rng.random() < 0.3, frame=rng.choice([24, 1560]),
                structure=rng.choice(["iid", "lowrank"]), q_gain=gain, lse=rng.random() < 0.5)


# ------------------------------------------------------------------------------------ inputs
def _workload(case):
    return wl.Workload(case.get("name", "drawn"), 50, n_heads=case["heads"], d_head=case["d_head"], T=_ints(case["T"]),
                       budget=_ints(case["budget"]), n_sink=case["sink"], n_recent=case["recent"], Lq=_ints(case["Lq"]),
                       d_hidden=case["hidden"], final=wl.FINAL_SIGMOID if case["sigmoid"] else wl.FINAL_NONE,
                       tokens_per_frame=case["frame"], structure=case["structure"])


def _randn(seed, *shape):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed & 0x7FFFFFFF)
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float32)


def _step_inputs(case, seed):
    w = _workload(case)
    data = wl.make_layer_device(w, seed=seed)
    if case["q_gain"] != 1.0:                       # peaked attention rows
        data["Q"] = (data["Q"].float() * case["q_gain"]).to(torch.bfloat16)
    return w, data


def _attn_inputs(case, seed):
    N, D, nB, nQ = case["heads"], case["d_head"], sum(_ints(case["B"])), sum(_ints(case["Lq"]))
    x = _randn(seed, 2 * nB + 3 * nQ, N, D)
    x[2 * (nB + nQ):] *= case["q_gain"]
    return [t.contiguous() for t in x.to(torch.bfloat16).split([nB, nB, nQ, nQ, nQ])]      # Kc, Vc, Kq, Vq, Q


def _cache_inputs(case, seed):
    N, D, nl = case["heads"], case["d_head"], case["layers"]
    d_in = 3 * N * D
    K = [_randn(seed * 131 + 4 * l + 1, case["capacity"], N, D).to(torch.bfloat16) for l in range(nl)]
    V = [_randn(seed * 131 + 4 * l + 2, case["capacity"], N, D).to(torch.bfloat16) for l in range(nl)]
    Kn = [_randn(seed * 131 + 4 * l + 3, case["chunk"], N, D).to(torch.bfloat16) for l in range(nl)]
    Vn = [_randn(seed * 131 + 4 * l + 4, case["chunk"], N, D).to(torch.bfloat16) for l in range(nl)]
    q = _randn(seed * 131 + 900, case["chunk"], N, D).to(torch.bfloat16)
    SL = 0.3 * _randn(seed * 131 + 901, case["capacity"])
    w1 = (_randn(seed * 131 + 902, PAPER_HIDDEN, d_in) / math.sqrt(d_in)).to(torch.bfloat16)
    b1 = (_randn(seed * 131 + 903, PAPER_HIDDEN) / math.sqrt(d_in)).to(torch.bfloat16)
    w2 = (_randn(seed * 131 + 904, PAPER_OUT, PAPER_HIDDEN) / math.sqrt(PAPER_HIDDEN)).to(torch.bfloat16)
    b2 = (_randn(seed * 131 + 905, PAPER_OUT) / math.sqrt(PAPER_HIDDEN)).to(torch.bfloat16)
    return K, V, Kn, Vn, q, SL, (w1, b1, w2, b2)


def _sse_inputs(case, seed):
    q = (2.0 * _randn(seed * 2 + 1, case["L"], case["heads"], 128)).to(torch.bfloat16)
    k = _randn(seed * 2 + 2, case["L"], case["heads"], 128).to(torch.bfloat16)
    return q, k


def _lse64(q, k, rows=2048):
    """Log-sum-exp of every row of q k^T / sqrt(128), [heads, L], in 64 bits."""
    out = torch.empty(q.shape[1], q.shape[0], dtype=torch.float64, device=q.device)
    for n in range(q.shape[1]):
        kn = k[:, n].double()
        for r in range(0, q.shape[0], rows):
            out[n, r:r + rows] = torch.logsumexp(q[r:r + rows, n].double() @ kn.T / math.sqrt(128), dim=1)
    return out


def prepare(case, seed):
    op = case["op"]
    if op in ("step", "step_indexed"):
        w, data = _step_inputs(case, seed)
        return op, Layer(w, data, want_lse=case["lse"], want_slc=True)
    if op == "attn":
        Kc, Vc, Kq, Vq, Q = _attn_inputs(case, seed)
        N, D = case["heads"], case["d_head"]
        shape = B.Shape(N, D, None, np.concatenate([[0], np.cumsum(_ints(case["Lq"]))]))
        cu_B = np.concatenate([[0], np.cumsum(_ints(case["B"]))])
        O = torch.empty_like(Q)
        LSE = torch.empty((N, Q.shape[0]), dtype=torch.float32, device="cuda") if case["lse"] else None
        ws = torch.zeros(B.pafu_workspace_bytes(shape), dtype=torch.uint8, device="cuda")
        return op, (Q, Kc, Vc, cu_B, Kq, Vq, shape, O, LSE, ws)
    if op == "cache_update":
        K, V, Kn, Vn, q, SL, weights = _cache_inputs(case, seed)
        cache = B.Cache(case["layers"], case["heads"], case["d_head"], case["capacity"], case["sink"])
        for l in range(case["layers"]):
            cache.Kb[0][l].copy_(K[l])
            cache.Vb[0][l].copy_(V[l])
        cache.SLb[0].copy_(SL)
        head = B.Head(*weights, act=B.ACT_SILU)
        shape = B.Shape(case["heads"], case["d_head"], [0, case["chunk"]], [0, case["chunk"]])
        ws = torch.zeros(B.pafu_workspace_bytes(shape, None, head), dtype=torch.uint8, device="cuda")
        return op, (cache, head, q, Kn, Vn, ws, case["capacity"], case["capacity"] - case["chunk"])
    if op == "sse":
        q, k = _sse_inputs(case, seed)
        L, N = case["L"], case["heads"]
        f32 = lambda *shape: torch.empty(*shape, dtype=torch.float32, device="cuda")
        lse = _lse64(q, k).float() if case["with_lse"] else None
        gmax, gavg = (f32(L), f32(L)) if case["pools"] else (None, None)
        ws = torch.zeros(B.pafu_sse_workspace_bytes(L, N, 128, case["block"]), dtype=torch.uint8, device="cuda")
        return op, (q, k, lse, case["block"], f32(L), f32(3, L), gmax, gavg, ws)
    raise KeyError(op)


# -------------------------------------------------------------------------------------- a pass
def run(state):
    op, s = state
    if op == "step":
        s.step()
        return [s.scores, s.idx, s.Kc, s.Vc, s.SLc, s.O] + ([s.LSE] if s.LSE is not None else [])
    if op == "step_indexed":
        s.step_indexed()
        return [s.scores, s.idx, s.O] + ([s.LSE] if s.LSE is not None else [])
    if op == "attn":
        Q, Kc, Vc, cu_B, Kq, Vq, shape, O, LSE, ws = s
        B.pafu_chunk_attn(Q, Kc, Vc, cu_B, Kq, Vq, shape, 0.0, O, LSE, ws)
        return [O] + ([LSE] if LSE is not None else [])
    if op == "cache_update":
        cache, head, q, Kn, Vn, ws, capacity, kept = s
        # the same full cache every time: the update reads buffer set 0 and writes set 1
        cache.c.T, cache.c.cur = capacity, 0
        B.pafu_cache_update(cache, head, q, Kn[-1], Vn[-1], Kn, Vn, ws)
        return [cache.idx[:kept], cache.SL] + cache.K + cache.V
    q, k, lse, block, out, comp, gmax, gavg, ws = s
    B.pafu_sse(q, k, lse, block, 0.0, out, comp, ws, gmax, gavg)
    return [out, comp] + ([gmax, gavg] if gmax is not None else [])


# ------------------------------------------------------------------------- bounds and tolerances
def work(case):
    op, N = case["op"], case["heads"]
    if op == "sse":
        L = case["L"]
        passes = 1 if case["with_lse"] else 2            # the row statistics need the logits once more
        return {"bytes": 2 * L * N * 256 + 16 * L + (4 * N * L if case["with_lse"] else 0) + (8 * L if case["pools"] else 0),
                "flops": passes * 256 * L * L * N}
    dm, row = N * case["d_head"], N * case["d_head"] * 2
    if op == "cache_update":
        kept, chunk = case["capacity"] - case["chunk"], case["chunk"]
        w = (PAPER_HIDDEN * 3 * dm + PAPER_OUT * PAPER_HIDDEN) * 2
        return {"bytes": case["layers"] * 2 * 2 * (kept + chunk) * row + chunk * row + w + 4 * (case["capacity"] + 2 * kept + chunk),
                "flops": 2 * chunk * 3 * dm * PAPER_HIDDEN}
    lqs = _ints(case["Lq"])
    nQ = sum(lqs)
    bs = _ints(case["B"]) if op == "attn" else tuple(min(b, t) for b, t in zip(_ints(case["budget"]), _ints(case["T"])))
    flops = sum(4 * lq * (b + lq) * dm for lq, b in zip(lqs, bs))
    lse = 4 * N * nQ if case["lse"] else 0
    if op == "attn":
        return {"bytes": (2 * sum(bs) + 4 * nQ) * row + lse, "flops": flops}
    nT, nB = sum(_ints(case["T"])), sum(bs)
    copies = 2 * nB * row + 4 * nB if op == "step" else 0                     # Kc, Vc, SLc written
    return {"bytes": (nT + nB + 4 * nQ) * row + copies + 4 * nT + 4 * nB + lse + 2 * case["hidden"] * (dm + 2),
            "flops": flops + 2 * nT * dm * case["hidden"]}


def tolerance(case):
    # bf16 probabilities and outputs: 2e-3 to 2.3e-3 against 64 bits; indices and copied rows are exact
    if case["op"] in ("step", "step_indexed", "attn"):
        return {"rel": 1e-2, "max": 0.05, "differ": 0.0}
    if case["op"] == "cache_update":                    # 32-bit sums of the chunk's scores (3e-6); the rest is copied
        return {"rel": 2e-5, "max": 2e-4, "differ": 0.0}
    return {"rel": 1e-5, "max": 1e-4}                   # probabilities exp(z - lse) of 32-bit logits: 1e-6 and less


# -------------------------------------------------------------------------------- 64-bit results
def _scores64(x, w1, b1, w2, b2, silu, sigmoid, rows=8192):
    w1, b1 = w1.double(), b1.double()
    w2, b2 = w2.double().mean(0), b2.double().mean()
    out = torch.empty(x[0].shape[0], dtype=torch.float64, device=w1.device)
    for r in range(0, out.shape[0], rows):
        h = torch.cat([p[r:r + rows].reshape(-1, w1.shape[1] // len(x)) for p in x], dim=1).double() @ w1.T + b1
        h = h * torch.sigmoid(h) if silu else torch.nn.functional.gelu(h)
        out[r:r + rows] = h @ w2 + b2
    return torch.sigmoid(out) if sigmoid else out


def _kept64(scores, n_sink, n_recent, budget):
    """Kept token indices; None where 32-bit scores could order the last kept token and the first
    dropped one the other way."""
    T = scores.shape[0]
    if T <= budget:
        return torch.arange(T, device=scores.device)
    nr = min(n_recent, budget)
    ns = min(n_sink, budget - nr)
    k = budget - ns - nr
    mid = scores[ns:T - nr]
    order = torch.argsort(mid, descending=True)
    if 0 < k < mid.shape[0] and float(mid[order[k - 1]] - mid[order[k]]) < 2e-6:
        return None
    top = ns + torch.sort(order[:k]).values
    return torch.cat([torch.arange(ns, device=top.device), top, torch.arange(T - nr, T, device=top.device)])


def _attn64(q, keys, values, rows=1024):
    """softmax(q k^T / sqrt(D)) v and the row log-sum-exps [heads, rows] of one stream."""
    N, D = q.shape[1:]
    o = torch.empty(q.shape, dtype=torch.float64, device=q.device)
    lse = torch.empty(N, q.shape[0], dtype=torch.float64, device=q.device)
    for n in range(N):
        kn = torch.cat([k[:, n] for k in keys]).double().T / math.sqrt(D)
        vn = torch.cat([v[:, n] for v in values]).double()
        for r in range(0, q.shape[0], rows):
            z = q[r:r + rows, n].double() @ kn
            l = torch.logsumexp(z, dim=1)
            o[r:r + rows, n] = torch.exp(z - l[:, None]) @ vn
            lse[n, r:r + rows] = l
    return o, lse


def exact(case, seed):
    with torch.no_grad():
        return _exact(case, seed)


def _exact(case, seed):
    op = case["op"]
    if op == "attn":
        Kc, Vc, Kq, Vq, Q = _attn_inputs(case, seed)
        lqs, bs = _ints(case["Lq"]), _ints(case["B"])
        got = [_attn64(q, (kc, kq), (vc, vq)) for q, kc, vc, kq, vq in zip(
            Q.split(lqs), Kc.split(bs), Vc.split(bs), Kq.split(lqs), Vq.split(lqs))]
        return [torch.cat([o for o, _ in got])] + ([torch.cat([l for _, l in got], dim=1)] if case["lse"] else [])
    if op == "cache_update":
        K, V, Kn, Vn, q, SL, weights = _cache_inputs(case, seed)
        idx = _kept64(SL, case["sink"], 0, case["capacity"] - case["chunk"])      # the list itself is 32-bit data
        new = _scores64([q, Kn[-1], Vn[-1]], *weights, silu=True, sigmoid=False)
        if idx is None:
            return [None, None] + [None] * (2 * case["layers"])
        roll = lambda old, add: torch.cat([old[idx], add])
        return ([idx.to(torch.int32), roll(SL.double(), new)] + [roll(K[l], Kn[l]) for l in range(case["layers"])] +
                [roll(V[l], Vn[l]) for l in range(case["layers"])])
    if op == "sse":
        return _sse64(case, seed)
    w, d = _step_inputs(case, seed)
    scores = _scores64([d["K"]], d["w1"], d["b1"], d["w2"], d["b2"], silu=False, sigmoid=case["sigmoid"])
    kept = [_kept64(s, w.n_sink, w.n_recent, b) for s, b in zip(scores.split(w.T), w.budget)]
    tail = 1 if case["lse"] else 0
    if any(k is None for k in kept):
        return [scores] + [None] * ((4 if op == "step" else 1) + 1 + tail)
    pick = lambda x: torch.cat([p[k] for p, k in zip(x.split(w.T), kept)])
    Kc, Vc, bs = pick(d["K"]), pick(d["V"]), [k.shape[0] for k in kept]
    got = [_attn64(q, (kc, kq), (vc, vq)) for q, kc, vc, kq, vq in zip(
        d["Q"].split(w.Lq), Kc.split(bs), Vc.split(bs), d["Kq"].split(w.Lq), d["Vq"].split(w.Lq))]
    copies = [Kc, Vc, pick(scores)] if op == "step" else []
    return ([scores, torch.cat(kept).to(torch.int32)] + copies + [torch.cat([o for o, _ in got])] +
            ([torch.cat([l for _, l in got], dim=1)] if tail else []))


def _sse64(case, seed):
    q, k = _sse_inputs(case, seed)
    L, N, LB = case["L"], case["heads"], case["block"]
    lse = _lse64(q, k)
    low, diag, up, avg, top = (torch.zeros(L, dtype=torch.float64, device=q.device) for _ in range(5))
    for n in range(N):
        kn = k[:, n].double().T / math.sqrt(128)
        best = torch.zeros(3, L, dtype=torch.float64, device=q.device)
        for b0 in range(0, L, LB):
            b1 = min(b0 + LB, L)
            for r in range(b0, b1, 2048):
                e = min(r + 2048, b1)
                P = torch.exp(q[r:e, n].double() @ kn - lse[n, r:e, None])
                m = P.max(0).values
                avg += P.sum(0) / (N * L)
                best[0, :b0] = torch.maximum(best[0, :b0], m[:b0])
                best[1, b0:b1] = torch.maximum(best[1, b0:b1], m[b0:b1])
                best[2, b1:] = torch.maximum(best[2, b1:], m[b1:])
        low += best[0] / N
        diag += best[1] / N
        up += best[2] / N
        top += best.max(0).values / N
    j = torch.arange(L, device=q.device)
    s = torch.where(j < LB, (diag + low) / 2, torch.where(j < L - LB, (up + diag + low) / 3, (diag + up) / 2))
    return [s, torch.stack([low, diag, up])] + ([top, avg] if case["pools"] else [])
