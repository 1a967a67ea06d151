"""GPU parity: every step of the CUDA path, called through the C ABI, against the CPU oracle
on the same seeded inputs.  Integer and byte results must be bit exact; scores and attention
outputs must agree within max-abs 2e-2 and mean-abs 2e-3 (bf16 inputs, fp32 accumulation)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2601_21896_b200 as pafu
from paper_2601_21896_b200 import workloads as wl
from paper_2601_21896_b200.harness import Layer, bf16_to_bits, to_device_bf16

pytestmark = pytest.mark.gpu

MAX_ABS, MEAN_ABS = 2e-2, 2e-3
# Beside the absolute bounds, an error bound relative to the size of the result: bf16 rounding of
# the output alone gives a relative Frobenius error of about 2^-9 / sqrt(3) = 1.1e-3, the bf16
# probabilities about as much again (2.0e-3 to 2.3e-3 is what the kernels show on every input),
# so 5e-3 leaves room and still rejects a result that is half a percent off when the values
# themselves are ~0.01 (near-uniform attention over thousands of keys).
REL_FRO = 5e-3


def close(got, want, what="", scaled=False):
    """The stated floating-point bounds (max-abs 2e-2, mean-abs 2e-3) plus the relative bound above.  `scaled`:
    the inputs were built to give outputs of magnitude up to ~4.5 (attention that picks single
    value rows); bf16 rounding of an output o alone is up to 2^-8 |o| = 1.8e-2 there, and the bf16
    probabilities add up to 2^-8 max|v|, so the absolute bounds grow with max|want|."""
    got = np.asarray(got, dtype=np.float64); want = np.asarray(want, dtype=np.float64)
    assert got.shape == want.shape, (got.shape, want.shape)
    if got.size == 0:
        return
    assert np.all(np.isfinite(got)), what
    err = np.abs(got - want)
    norm = np.sqrt((want * want).sum())
    rel = np.sqrt((err * err).sum()) / norm if norm > 1e-30 else 0.0
    print("%s: max-abs %.3e mean-abs %.3e rel-fro %.3e (max|want| %.3g)" % (what, err.max(), err.mean(), rel,
                                                                             np.abs(want).max()))
    grow = max(1.0, np.abs(want).max()) if scaled else 1.0
    assert err.max() <= MAX_ABS * grow, (what, err.max(), np.unravel_index(err.argmax(), err.shape))
    assert err.mean() <= MEAN_ABS * grow, (what, err.mean())
    assert rel <= REL_FRO, (what, rel)


def oracle_scores(w, d):
    return oracle.score(d["K"].reshape(d["K"].shape[0], -1), d["w1"], d["b1"], d["w2"], d["b2"],
                        w.act, w.final)


def oracle_select_streams(scores, w):
    cuT = w.cu("T")
    return [oracle.select(scores[cuT[s]:cuT[s + 1]], w.n_sink, w.n_recent, w.budget[s])
            for s in range(w.n_streams)]


def oracle_attn_streams(w, d, Kc_bits, Vc_bits, cu_B, rows=None):
    cuQ = w.cu("Lq")
    outs = []
    for s in range(w.n_streams):
        q = d["Q"][cuQ[s]:cuQ[s + 1]]
        r = None if rows is None else rows[s]
        O, L = oracle.attention(q, Kc_bits[cu_B[s]:cu_B[s + 1]], Vc_bits[cu_B[s]:cu_B[s + 1]],
                                d["Kq"][cuQ[s]:cuQ[s + 1]], d["Vq"][cuQ[s]:cuQ[s + 1]], rows=r)
        outs.append((O, L))
    return outs


SMALL = [wl.tiny(), wl.small_ragged(2, 128), wl.small_ragged(3, 64)]


# --------------------------------------------------------------------------------- score
@pytest.mark.parametrize("w", SMALL, ids=lambda w: "%s-d%d" % (w.name, w.d_head))
def test_score_matches_oracle(w):
    d = wl.make_layer(w)
    L = Layer(w, d)
    L.score()
    L.check_status()
    close(L.scores[: L.nT].cpu().numpy(), oracle_scores(w, d), "score")


@pytest.mark.parametrize("act,final,d_out,d_hidden,n", [
    (wl.ACT_SILU, wl.FINAL_NONE, 12, 1024, 300),     # the paper's S-MLP widths (Appendix A)
    (wl.ACT_GELU, wl.FINAL_SIGMOID, 1, 32, 129),
    (wl.ACT_GELU, wl.FINAL_NONE, 3, 272, 1),
    (wl.ACT_SILU, wl.FINAL_SIGMOID, 1, 256, 517),
])
def test_score_head_variants(act, final, d_out, d_hidden, n):
    rng = np.random.default_rng(5)
    d_in = 384
    bits = lambda shape, s=1.0: wl.f32_to_bf16_bits((rng.standard_normal(shape) * s).astype(np.float32))
    X = bits((n, d_in)); w1 = bits((d_hidden, d_in), d_in ** -0.5); b1 = bits((d_hidden,), 0.3)
    w2 = bits((d_out, d_hidden), d_hidden ** -0.5); b2 = bits((d_out,), 0.3)
    for use_bias in (True, False):
        dev = [to_device_bf16(a) for a in (X, w1, b1, w2, b2)]
        head = pafu.Head(dev[1], dev[2] if use_bias else None, dev[3], dev[4] if use_bias else None,
                         act, final)
        shape = pafu.Shape(3, 128, [0, n], [0, 1])
        ws = torch.zeros(pafu.pafu_workspace_bytes(shape, None, head), dtype=torch.uint8, device="cuda")
        out = torch.full((n,), float("nan"), device="cuda")
        pafu.pafu_score(head, dev[0], out, ws)
        assert pafu.pafu_workspace_status(ws) == 0
        want = oracle.score(X, w1, b1 if use_bias else None, w2, b2 if use_bias else None, act, final)
        close(out.cpu().numpy(), want, "score variant")


@pytest.mark.parametrize("d_part,d_hidden,d_out,act,n,ld_extra", [
    (1536, 1024, 12, wl.ACT_SILU, 4680, 0),    # the paper's S-MLP on one 3-frame chunk (Sec. 3.3, Appendix A)
    (128, 64, 1, wl.ACT_GELU, 301, 64),        # rows wider than the features used, ragged last tile
    (64, 272, 3, wl.ACT_SILU, 1, 0),
])
def test_score_qkv_matches_oracle_on_concatenated_rows(d_part, d_hidden, d_out, act, n, ld_extra):
    """x_t = [q_t, k_t, v_t] read from three matrices in place equals the plain head applied to
    the concatenated rows (the oracle sees only the concatenation)."""
    rng = np.random.default_rng(11)
    d_in = 3 * d_part
    ld = d_part + ld_extra
    bits = lambda shape, s=1.0: wl.f32_to_bf16_bits((rng.standard_normal(shape) * s).astype(np.float32))
    Q, K, V = bits((n, ld)), bits((n, ld)), bits((n, ld))
    w1 = bits((d_hidden, d_in), d_in ** -0.5); b1 = bits((d_hidden,), 0.3)
    w2 = bits((d_out, d_hidden), d_hidden ** -0.5); b2 = bits((d_out,), 0.3)
    dev = [to_device_bf16(a) for a in (Q, K, V, w1, b1, w2, b2)]
    head = pafu.Head(dev[3], dev[4], dev[5], dev[6], act, wl.FINAL_NONE)
    shape = pafu.Shape(3, 128, [0, n], [0, 1])
    ws = torch.zeros(pafu.pafu_workspace_bytes(shape, None, head), dtype=torch.uint8, device="cuda")
    out = torch.full((n,), float("nan"), device="cuda")
    pafu.pafu_score_qkv(head, dev[0], dev[1], dev[2], out, ws, ld=ld)
    assert pafu.pafu_workspace_status(ws) == 0
    X = np.ascontiguousarray(np.concatenate([Q[:, :d_part], K[:, :d_part], V[:, :d_part]], axis=1))
    want = oracle.score(X, w1, b1, w2, b2, act, wl.FINAL_NONE)
    close(out.cpu().numpy(), want, "score qkv")
    # and the one-matrix entry on the same concatenation gives the same bits
    out1 = torch.full((n,), float("nan"), device="cuda")
    pafu.pafu_score(head, to_device_bf16(X), out1, ws)
    assert torch.equal(out, out1)


# -------------------------------------------------------------------------------- select
@pytest.mark.parametrize("kind", ["normal", "ties", "equal", "saturated", "heavy", "signed_zero"])
def test_select_bit_exact(kind):
    cases = [((512,), 4, 64, (128,)), ((1000, 37, 2048, 5), 3, 10, (500, 20, 1024, 9)),
             ((4097,), 0, 0, (1,)), ((4097,), 0, 0, (4096,)), ((3000,), 100, 200, (250,)),
             ((3000,), 5000, 0, (1000,)), ((1, 2, 3), 1, 1, (0, 1, 2)), ((28080,), 1560, 4680, (14040,)),
             ((93600,), 1560, 4680, (9360,)),
             # longer streams, selected by clusters of eight
             ((53248 + 30,), 10, 20, (20000,)), ((53249 + 30,), 10, 20, (20000,)), ((106496 + 7,), 3, 4, (106000,)),
             # shares that look near the k-th largest candidate only; and long and short streams in one call
             ((106497 + 7,), 3, 4, (555,)), ((200000,), 1560, 4680, (20000,)),
             ((1000, 40000, 90000, 200000, 64), 10, 100, (500, 9000, 30000, 50000, 64))]
    for ci, (T, ns, nr, Bs) in enumerate(cases):
        n = len(T)
        cuT = np.concatenate([[0], np.cumsum(T)])
        s = wl.random_scores(int(cuT[-1]), seed=ci, kind=kind, tag=ci)
        if kind == "heavy":
            s[::97] = np.nan; s[5::101] = np.inf; s[7::103] = -np.inf
        shape = pafu.Shape(1, 64, cuT, None)
        pol = pafu.make_policy(ns, nr, list(Bs), n)
        cu_B = pafu.pafu_kept_counts(shape, pol)
        idx = torch.full((max(int(cu_B[-1]), 1),), -1, dtype=torch.int32, device="cuda")
        pafu.pafu_select(torch.from_numpy(s).cuda(), shape, pol, idx)
        got = idx.cpu().numpy()
        for st in range(n):
            want = oracle.select(s[cuT[st]:cuT[st + 1]], ns, nr, Bs[st])
            assert cu_B[st + 1] - cu_B[st] == len(want)
            assert np.array_equal(got[cu_B[st]:cu_B[st + 1]], want), (kind, ci, st)


@pytest.mark.parametrize("kind", ["steps", "equal", "outlier", "two_values", "one_bin_256", "one_bin_257", "denormal", "infinite"])
def test_select_histogram_routes(kind):
    """Sizes around what one warp, one block and 1, 2, 4, 8 CTAs take, with scores that spread over the value histogram, that
    fall into one bin of it (as many as are ranked directly, and one more), and that leave it no finite range."""
    rng = np.random.default_rng(11)
    for M in (1, 2, 31, 33, 255, 257, 600, 1024, 1025, 4096, 4097, 8193, 16385, 33000):
        s = rng.standard_normal(M + 5).astype(np.float32)
        if kind == "equal":
            s[:] = 0.25
        elif kind == "outlier":
            s[::256] = 1e30
        elif kind == "two_values":
            s = np.where(s > 0, np.float32(1), np.float32(-1))
        elif kind.startswith("one_bin"):
            s = (100 * np.sign(s) + s).astype(np.float32)
            n = min(int(kind[-3:]), M)
            s[3 + rng.permutation(M)[:n]] = (0.01 * rng.standard_normal(n)).astype(np.float32)
        elif kind == "denormal":
            s *= np.float32(1e-44)
        elif kind == "infinite":
            s = rng.choice(np.array([np.inf, -np.inf, np.nan, 3.4e38, -3.4e38], np.float32), M + 5)
        for k in sorted({1, M // 3, M // 2, M - 1} - {0}):
            shape = pafu.Shape(1, 64, [0, M + 5], None)
            idx = torch.full((k + 5,), -1, dtype=torch.int32, device="cuda")
            pafu.pafu_select(torch.from_numpy(s).cuda(), shape, pafu.make_policy(3, 2, [k + 5], 1), idx)
            assert np.array_equal(idx.cpu().numpy(), oracle.select(s, 3, 2, k + 5)), (kind, M, k)


@pytest.mark.parametrize("M", [8 * 11264, 8 * 11264 + 1, 200000, 360448])
@pytest.mark.parametrize("kind", ["normal", "outlier", "frames", "equal", "one_bin", "one_bin_in_one_cta", "one_bin_too_many", "extremes"])
def test_select_long_shares(M, kind):
    """Shares around the length from which the steps lie near the k-th largest candidate, and the longest one; one bin with as many
    candidates as are ranked directly, spread over the CTAs or all in one's, and one more; k in the tails."""
    rng = np.random.default_rng(M)
    s = rng.standard_normal(M).astype(np.float32)
    ks = [1, M // 700, M // 2, M - M // 50, M - 1]
    if kind == "outlier":
        s[::257] = 1e30
    elif kind == "frames":
        s = (0.1 * s + np.repeat(rng.standard_normal(M // 1560 + 1), 1560)[:M]).astype(np.float32)
    elif kind == "equal":
        s[:] = -3.5
    elif kind == "extremes":
        s = rng.choice(np.array([np.inf, -np.inf, np.nan, 3.4e38, -3.4e38, 1e-44, -1e-44, 0.0, -0.0], np.float32), M)
    elif kind.startswith("one_bin"):
        per_cta = (-(-M // 8) + 31) // 32 * 32
        n = max(256, min(1024, per_cta // 32)) + (kind == "one_bin_too_many")
        s = (100 * np.sign(s) + s).astype(np.float32)
        at = rng.permutation(M)[:n] if kind != "one_bin_in_one_cta" else per_cta + rng.permutation(per_cta)[:n]
        s[at] = (0.001 * rng.standard_normal(n)).astype(np.float32)
        above = int((s > 50).sum())
        ks = [above, above + 1, above + n // 2, above + n, above + n + 1]
    d = torch.from_numpy(s).cuda()
    for k in ks:
        idx = torch.full((k,), -1, dtype=torch.int32, device="cuda")
        pafu.pafu_select(d, pafu.Shape(1, 64, [0, M], None), pafu.make_policy(0, 0, [k], 1), idx)
        assert np.array_equal(idx.cpu().numpy(), oracle.select(s, 0, 0, k)), (kind, M, k)


# ------------------------------------------------------------------------------- compact
@pytest.mark.parametrize("w", SMALL + [wl.Workload("odd_dm", 7, 5, 8, (77, 9), (30, 9), 2, 3, (4, 4), 32)],
                         ids=lambda w: "%s-dm%d" % (w.name, w.d_model))
def test_compact_bit_exact(w):
    d = wl.make_layer(w, tensors=("K", "V"))
    rng = np.random.default_rng(3)
    cuT = w.cu("T"); cuB = w.cu("B")
    idx_np = np.concatenate([np.sort(rng.choice(w.T[s], size=cuB[s + 1] - cuB[s], replace=False))
                             for s in range(w.n_streams)]).astype(np.int32)
    SL = rng.standard_normal(int(cuT[-1])).astype(np.float32)
    shape = pafu.Shape(w.n_heads, w.d_head, cuT, None)
    pol = pafu.make_policy(w.n_sink, w.n_recent, list(w.budget), w.n_streams)
    K, V = to_device_bf16(d["K"]), to_device_bf16(d["V"])
    nB = int(cuB[-1])
    Kc = torch.zeros((nB, w.n_heads, w.d_head), dtype=torch.bfloat16, device="cuda")
    Vc = torch.zeros_like(Kc)
    SLc = torch.zeros(nB, device="cuda")
    pafu.pafu_compact(K, V, torch.from_numpy(SL).cuda(), torch.from_numpy(idx_np).cuda(), shape, pol,
                      Kc, Vc, SLc)
    for s in range(w.n_streams):
        i = idx_np[cuB[s]:cuB[s + 1]]
        assert np.array_equal(bf16_to_bits(Kc)[cuB[s]:cuB[s + 1]], oracle.compact(d["K"][cuT[s]:cuT[s + 1]], i))
        assert np.array_equal(bf16_to_bits(Vc)[cuB[s]:cuB[s + 1]], oracle.compact(d["V"][cuT[s]:cuT[s + 1]], i))
        assert np.array_equal(SLc.cpu().numpy()[cuB[s]:cuB[s + 1]], oracle.compact(SL[cuT[s]:cuT[s + 1]], i))
    # inputs untouched
    assert np.array_equal(bf16_to_bits(K), d["K"]) and np.array_equal(bf16_to_bits(V), d["V"])


@pytest.mark.parametrize("d_head,n_heads,T,B", [
    (64, 1, (47000,), (45000,)),                            # rows of 8 pieces: 12 at once, one selecting cluster
    (64, 1, (9000, 700, 9, 40000), (9000, 650, 0, 39999)),  # four streams, one kept whole, one empty: rows are claimed
    (64, 3, (12000,), (11111,)),                            # 24 pieces, the last group short
    (128, 6, (11000,), (10700,)),                           # 96 pieces: two rows at once
    (128, 6, (11000,), (10600,)),                           # fewer than three rows a warp: one at a time
], ids=lambda v: str(v) if isinstance(v, int) else "x".join(map(str, v)))
def test_gather_of_narrow_rows(d_head, n_heads, T, B):
    """The row gather's groups of rows, behind the selection inside a step and by itself: every kept row and score is a copy."""
    w = wl.Workload("narrow", 8, n_heads, d_head, T, B, 7, 9, (64,) * len(T), 32)
    L = Layer(w, wl.make_layer_device(w, seed=3))
    L.step(); L.check_status()
    cuT, cuB = w.cu("T"), L.cu_B
    idx = torch.cat([L.idx[cuB[s]:cuB[s + 1]].long() + int(cuT[s]) for s in range(len(T))])
    for again in range(2):
        assert torch.equal(L.Kc[:L.nB], L.K[idx]) and torch.equal(L.Vc[:L.nB], L.V[idx])
        assert torch.equal(L.SLc[:L.nB], L.scores[idx])
        L.Kc.zero_(); L.Vc.zero_(); L.SLc.zero_()
        L.compact()


@pytest.mark.parametrize("d_head,n_heads,T,B,sink,recent,slc", [
    (64, 1, (3, 1), (2, 1), 0, 0, True),                        # smaller than a warp; a stream kept whole
    (64, 2, (1100, 40, 9), (1, 40, 0), 0, 0, False),            # one row, everything, nothing; no salience list
    (64, 3, (1024 + 30, 1025 + 30), (300, 30), 10, 20, True),   # candidates around a small block's; no top-k row at all
    (128, 2, (4096 + 7, 2000), (4000, 1999), 3, 4, True),       # the most one CTA selects
    (128, 2, (4097 + 7, 2000), (4000, 1999), 3, 4, True),       # one more: two launches
    (128, 3, (30000,), (29000,), 27000, 100, True),             # 89 MB: two launches
    (128, 3, (13000,), (12600,), 12000, 100, True),             # few candidates, many rows: 38.7 MB in and out in one launch
    (64, 2, (36000,) + (60, 9) * 15 + (100,), (36000,) + (30, 0) * 15 + (99,), 3, 4, True),   # one stream kept whole beside 31 short ones
], ids=lambda v: str(v) if not isinstance(v, tuple) else "x".join(map(str, v)))
def test_small_step_selects_and_copies_in_one_launch(d_head, n_heads, T, B, sink, recent, slc):
    """The same indices, rows and scores as the separate calls."""
    w = wl.Workload("small", 9, n_heads, d_head, T, B, sink, recent, (64,) * len(T), 32)
    d = wl.make_layer_device(w, seed=5)
    A, S = Layer(w, d, want_slc=slc), Layer(w, d, want_slc=slc)
    for t in (A.idx, S.idx):
        t.fill_(-1)
    for t in (A.Kc, A.Vc, S.Kc, S.Vc):
        t.zero_()
    A.step(); A.check_status()
    S.score(); S.select(); S.compact(); S.attn(); S.check_status()
    assert torch.equal(A.idx, S.idx) and torch.equal(A.Kc, S.Kc) and torch.equal(A.Vc, S.Vc)
    assert not slc or torch.equal(A.SLc[:A.nB], S.SLc[:S.nB])
    assert torch.equal(A.O, S.O)


@pytest.mark.parametrize("kind", ["equal", "two_values", "not_finite"])
@pytest.mark.parametrize("T,B", [((700, 333), (300, 100)), ((4096,), (1500,)), ((4000, 30), (3999, 7))], ids=str)
def test_small_step_with_ties_and_scores_that_are_not_finite(T, B, kind):
    """Bins that have to be narrowed down, in the launch that selects and copies: the oracle's indices on its scores, and copies."""
    w = wl.Workload("tied", 9, 2, 64, T, B, 3, 5, (64,) * len(T), 32, final=wl.FINAL_SIGMOID if kind == "two_values" else wl.FINAL_NONE)
    d = wl.make_layer_device(w, seed=5)
    if kind == "equal":
        d["w2"] = torch.zeros_like(d["w2"])
    elif kind == "two_values":
        d["w2"] = d["w2"] * 8192.0                               # the sigmoid saturates
    else:
        d["w1"][:, 0] = 3.0e38; d["w2"] = d["w2"].abs()          # infinities, NaN (0 x -inf) and zeros of both signs
    L = Layer(w, d)
    L.step(); L.check_status()
    scores, cuT, cuB = L.scores.cpu().numpy(), w.cu("T"), L.cu_B
    if kind == "two_values":
        assert np.mean((scores[:cuT[-1]] == 0) | (scores[:cuT[-1]] == 1)) > 0.9
    elif kind == "not_finite":
        assert 0.1 < np.mean(~np.isfinite(scores[:cuT[-1]])) < 0.9
    for s in range(len(T)):
        ids = oracle.select(scores[cuT[s]:cuT[s + 1]], 3, 5, B[s])
        assert np.array_equal(L.idx[cuB[s]:cuB[s + 1]].cpu().numpy(), ids)
        rows = torch.from_numpy(ids.astype(np.int64)).cuda() + int(cuT[s])
        for got, want in ((L.Kc, L.K), (L.Vc, L.V), (L.SLc, L.scores)):
            bits = torch.int16 if got.dtype == torch.bfloat16 else torch.int32
            assert torch.equal(got[cuB[s]:cuB[s + 1]].view(bits), want[rows].view(bits))


# ----------------------------------------------------------------------------- attention
@pytest.mark.parametrize("w", SMALL, ids=lambda w: "%s-d%d" % (w.name, w.d_head))
def test_attention_matches_oracle_everywhere(w):
    d = wl.make_layer(w)
    L = Layer(w, d)
    # retained cache = the oracle's own selection, so attention is tested on its own
    sc = oracle_scores(w, d)
    idx = oracle_select_streams(sc, w)
    cuT, cuB = w.cu("T"), L.cu_B
    Kc = np.concatenate([oracle.compact(d["K"][cuT[s]:cuT[s + 1]], idx[s]) for s in range(w.n_streams)])
    Vc = np.concatenate([oracle.compact(d["V"][cuT[s]:cuT[s + 1]], idx[s]) for s in range(w.n_streams)])
    L.Kc.copy_(to_device_bf16(Kc)); L.Vc.copy_(to_device_bf16(Vc))
    L.O.fill_(float("nan")); L.LSE.fill_(float("nan"))
    L.attn()
    L.check_status()
    got = wl.bf16_bits_to_f32(bf16_to_bits(L.O))
    lse = L.LSE.cpu().numpy()
    cuQ = w.cu("Lq")
    for s, (O, Ls) in enumerate(oracle_attn_streams(w, d, Kc, Vc, cuB)):
        close(got[cuQ[s]:cuQ[s + 1]], O, "attn O stream %d" % s)
        close(lse[:, cuQ[s]:cuQ[s + 1]], Ls, "attn LSE stream %d" % s)


def test_attention_segment_edge_cases():
    # no retained cache / no chunk segment / one key / lengths around the tile sizes
    rng = np.random.default_rng(9)
    N, D = 2, 128
    for (Lq, nB, chunk) in [(1, 0, True), (5, 1, False), (64, 64, True), (65, 127, True),
                            (129, 128, False), (130, 257, True), (3, 0, False)]:
        bits = lambda n: wl.f32_to_bf16_bits(rng.standard_normal((n, N, D)).astype(np.float32))
        Q, Kc, Vc, Kq, Vq = bits(Lq), bits(nB), bits(nB), bits(Lq), bits(Lq)
        shape = pafu.Shape(N, D, None, [0, Lq])
        dv = lambda a: to_device_bf16(a) if a.shape[0] else torch.zeros((1, N, D), dtype=torch.bfloat16, device="cuda")
        O = torch.full((Lq, N, D), float("nan"), dtype=torch.bfloat16, device="cuda")
        LSE = torch.full((N, Lq), float("nan"), device="cuda")
        ws = torch.zeros(max(pafu.pafu_workspace_bytes(shape), 256), dtype=torch.uint8, device="cuda")
        pafu.pafu_chunk_attn(dv(Q), dv(Kc), dv(Vc), [0, nB], dv(Kq) if chunk else None,
                             dv(Vq) if chunk else None, shape, 0.0, O, LSE, ws)
        assert pafu.pafu_workspace_status(ws) == 0
        want, wl_ = oracle.attention(Q, Kc, Vc, Kq if chunk else None, Vq if chunk else None)
        got = wl.bf16_bits_to_f32(bf16_to_bits(O))
        if nB == 0 and not chunk:
            assert np.all(got == 0) and np.all(np.isneginf(LSE.cpu().numpy()))
        else:
            close(got, want, "edge O %s" % ((Lq, nB, chunk),))
            close(LSE.cpu().numpy(), wl_, "edge LSE")


@pytest.mark.parametrize("kind", ["one_run", "runs", "steps_of_two", "unsorted", "ragged_run"])
def test_indexed_attention_takes_runs_tiled(kind):
    """Tiles of neighbouring cache rows are loaded tiled, all others row by row: the same bits as on gathered rows."""
    g = torch.Generator(device="cuda"); g.manual_seed(7)
    N, D, Lq = 3, 128, (200, 300)
    T = (900, 700)
    rn = lambda n: torch.randn(n, N, D, generator=g, device="cuda").to(torch.bfloat16)
    K, V, Q, Kq, Vq = rn(sum(T)), rn(sum(T)), rn(sum(Lq)), rn(sum(Lq)), rn(sum(Lq))
    ar = lambda a, b: torch.arange(a, b, device="cuda")
    lists = []
    for t in T:
        lists.append({"one_run": ar(37, 37 + 512), "runs": torch.cat([ar(0, 100), ar(130, 400), ar(401, 430)]),
                      "steps_of_two": ar(0, 256) * 2, "unsorted": torch.cat([ar(300, 428), ar(0, 64).flip(0), ar(64, 128)]),
                      "ragged_run": ar(t - 421, t)}[kind])
    cu_B = np.concatenate([[0], np.cumsum([len(i) for i in lists])])
    idx = torch.cat(lists).to(torch.int32)
    rows = torch.cat([lists[0], lists[1] + T[0]])
    shape = pafu.Shape(N, D, np.concatenate([[0], np.cumsum(T)]), np.concatenate([[0], np.cumsum(Lq)]))
    ws = torch.zeros(pafu.pafu_workspace_bytes(shape), dtype=torch.uint8, device="cuda")
    out = []
    for indexed in (False, True):
        O, LSE = torch.zeros_like(Q), torch.zeros(N, sum(Lq), device="cuda")
        if indexed:
            pafu.pafu_chunk_attn_indexed(Q, K, V, idx, cu_B, Kq, Vq, shape, 0.0, O, LSE, ws)
        else:
            pafu.pafu_chunk_attn(Q, K[rows].contiguous(), V[rows].contiguous(), cu_B, Kq, Vq, shape, 0.0, O, LSE, ws)
        assert pafu.pafu_workspace_status(ws) == 0
        out.append((O, LSE))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])


# ---------------------------------- peaked attention: the running maximum has to move (Sec. 3.2)
def _attention_all_entry_points(d, N, D, Lq, nB, what, seed=0):
    """One set of inputs through pafu_chunk_attn, pafu_chunk_attn_indexed (the retained rows
    scattered through a larger cache) and pafu_chunk_attn_noalloc, each element-wise against the
    oracle.  Returns the path counters of the pafu_chunk_attn launch."""
    want_O, want_lse = oracle.attention(d["Q"], d["Kc"], d["Vc"], d["Kq"], d["Vq"])
    dQ, dKc, dVc, dKq, dVq = [to_device_bf16(d[k]) for k in ("Q", "Kc", "Vc", "Kq", "Vq")]
    shape = pafu.Shape(N, D, None, [0, Lq])
    ws = torch.zeros(pafu.pafu_workspace_bytes(shape), dtype=torch.uint8, device="cuda")

    def fresh():
        return (torch.full((Lq, N, D), float("nan"), dtype=torch.bfloat16, device="cuda"),
                torch.full((N, Lq), float("nan"), device="cuda"))

    def check(O, LSE, name):
        close(wl.bf16_bits_to_f32(bf16_to_bits(O)), want_O, "%s %s O" % (what, name), scaled=True)
        close(LSE.cpu().numpy(), want_lse, "%s %s LSE" % (what, name))

    O, LSE = fresh()
    pafu.pafu_chunk_attn(dQ, dKc, dVc, [0, nB], dKq, dVq, shape, 0.0, O, LSE, ws)
    assert pafu.pafu_workspace_status(ws) == 0
    counts = pafu.pafu_workspace_counters(ws)
    check(O, LSE, "chunk_attn")
    # the same retained rows reached through an index list into a cache 1.5 x as long
    rng = np.random.default_rng(seed + 1)
    T = nB + nB // 2 + 7
    idx = np.sort(rng.choice(T, size=nB, replace=False)).astype(np.int32)
    Kraw = wl.f32_to_bf16_bits(rng.standard_normal((T, N, D)).astype(np.float32)); Vraw = Kraw.copy()
    Kraw[idx] = d["Kc"]; Vraw[idx] = d["Vc"]
    O2, LSE2 = fresh()
    pafu.pafu_chunk_attn_indexed(dQ, to_device_bf16(Kraw), to_device_bf16(Vraw), torch.from_numpy(idx).cuda(),
                                 [0, nB], dKq, dVq, pafu.Shape(N, D, [0, T], [0, Lq]), 0.0, O2, LSE2, ws)
    assert pafu.pafu_workspace_status(ws) == 0
    check(O2, LSE2, "indexed")
    assert torch.equal(O.view(torch.int16), O2.view(torch.int16)) and torch.equal(LSE, LSE2)
    O3, LSE3 = fresh()
    pafu.pafu_chunk_attn_noalloc(dQ, dKc, dVc, [0, nB], dKq, dVq, shape, 0.0, O3, LSE3)
    torch.cuda.synchronize()
    check(O3, LSE3, "noalloc")
    return counts


# (heads, chunk queries, retained keys): "short" gives every CTA a run of about two key tiles and
# splits every item over dozens of CTAs (the merge sees many pieces); "long" gives runs of about
# ten tiles (the in-kernel rescale has tiles before and after it).  Both have a ragged last query
# block, a ragged last retained tile and a ragged last chunk tile.
PEAKED_SIZES = {"short": (2, 600, 3017), "long": (2, 770, 12013)}


@pytest.mark.parametrize("size", ["short", "long"])
@pytest.mark.parametrize("q_scale", [4.0, 8.0, 16.0, 300.0])
def test_attention_scaled_logits(size, q_scale):
    N, Lq, nB = PEAKED_SIZES[size]
    d = wl.peaked_attention_inputs("scaled_q", N, 128, Lq, nB, seed=int(q_scale), q_scale=q_scale)
    c = _attention_all_entry_points(d, N, 128, Lq, nB, "Q x %g %s" % (q_scale, size))
    print("path counters (first/ragged exact, sum-triggered exact, rescales):", c.tolist())
    if q_scale >= 16.0 and size == "long":
        assert c[1] > 0 and c[2] > 0      # the input did reach the rescale path


@pytest.mark.parametrize("size", ["short", "long"])
@pytest.mark.parametrize("rise", [0.2, 3.0, 15.0, -0.2, -3.0, -15.0])
def test_attention_rising_and_falling_logits(size, rise):
    """Logits that rise along the key axis by `rise` nats per 64-key tile: gently (the running
    maximum goes stale but stays usable for dozens of tiles), by a few nats (a rescale every few
    tiles), steeply (every tile after a run's first is rescaled); and the mirror images, where the
    first tile holds the maximum for good."""
    N, Lq, nB = PEAKED_SIZES[size]
    d = wl.peaked_attention_inputs("ramp", N, 128, Lq, nB, seed=7, rise_per_tile=rise, varied_rows=(abs(rise) == 3.0))
    c = _attention_all_entry_points(d, N, 128, Lq, nB, "ramp %+g %s" % (rise, size))
    print("path counters:", c.tolist())
    if rise >= 3.0:
        assert c[2] > 0
    if rise == 15.0 and size == "long":
        n_tiles_rows = 2 * ((Lq + 127) // 128) * ((nB + 63) // 64 + (Lq + 63) // 64) * 4
        assert c[2] > n_tiles_rows // 2, (c.tolist(), n_tiles_rows)     # most (warp, tile) pairs rescale


def _spike_positions(size):
    N, Lq, nB = PEAKED_SIZES[size]
    mid = (nB // 2 // 64) * 64
    named = {"first_tile": [5], "middle_tile": [mid + 31], "ragged_retained_tile": [nB - 2], "chunk_segment": [nB + 17],
             "last_chunk_key": [nB + Lq - 1],
             # a weaker spike early, stronger ones later: pieces of one item whose maxima differ by tens of nats
             "three_rising": [70, mid + 3, nB + Lq - 40],
             "two_falling_in_strength": [nB + 100, 9]}
    # and one spike in each of twelve consecutive tiles: whatever the cut between CTAs, some land on a
    # run's first tile, some on its last, some on the last tile of a piece that another CTA continues
    for k in range(12):
        named["tile_%d" % k] = [mid + 64 * k + (17 * k) % 64]
    return named


@pytest.mark.parametrize("size", ["short", "long"])
@pytest.mark.parametrize("where", sorted(_spike_positions("short")))
def test_attention_dominating_keys(size, where):
    if size == "long" and where.startswith("tile_") and int(where[5:]) % 4 != 0:
        pytest.skip("the long size takes every fourth of the consecutive-tile positions")
    N, Lq, nB = PEAKED_SIZES[size]
    pos = _spike_positions(size)[where]      # a spike listed later is stronger (see the generator)
    d = wl.peaked_attention_inputs("spike", N, 128, Lq, nB, seed=3, spike_pos=pos, varied_rows=True)
    c = _attention_all_entry_points(d, N, 128, Lq, nB, "spike %s %s" % (where, size))
    print("path counters:", c.tolist())


@pytest.mark.parametrize("size", ["short", "long"])
def test_attention_run_opening_on_tiny_logits(size):
    """Every third key tile lies ~56 nats below the rest: a run that opens on one starts from a
    maximum far too small, the next tile's row sums overflow the fast path's range (2^16, or
    infinity) and the tile must be redone exactly and the accumulator rescaled by ~e^-56."""
    N, Lq, nB = PEAKED_SIZES[size]
    d = wl.peaked_attention_inputs("tiny_tiles", N, 128, Lq, nB, seed=5)
    c = _attention_all_entry_points(d, N, 128, Lq, nB, "tiny tiles %s" % size)
    print("path counters:", c.tolist())
    assert c[1] > 0 and c[2] > 0


@pytest.mark.parametrize("size", ["short", "long"])
def test_path_counters_stay_at_zero_on_ordinary_logits(size):
    """The control for the tests above: on N(0, 1) logits no row sum outgrows the running maximum (2^16 would take a logit
    11 nats above the opening tile's maximum) and nothing is rescaled, however short the runs are."""
    N, Lq, nB = PEAKED_SIZES[size]
    c = _attention_all_entry_points(wl.peaked_attention_inputs("scaled_q", N, 128, Lq, nB, seed=9, q_scale=1.0), N, 128, Lq, nB, "control")
    assert c[0] > 0 and c[1] == 0 and c[2] == 0, c.tolist()


@pytest.mark.parametrize("N,D,Lq,nB,run", [
    (2, 64, 64, 128, 1), (2, 128, 100, 300, 1),                  # one or two tiles a CTA at the finest: whole, or single tiles
    (4, 128, 600, 2000, 3), (4, 64, 600, 2000, 3),               # shares of three tiles
    (120, 128, 256, 300, 5), (140, 64, 256, 448, 6), (140, 128, 256, 448, 6),   # whole items of 9 and 11 tiles
    (8, 128, 600, 2000, 7),                                      # shares of six and a half
])
@pytest.mark.parametrize("q_scale", [1.0, 2.0, 4.0])
def test_attention_error_is_no_larger_than_in_pieces(N, D, Lq, nB, run, q_scale):
    """However a small problem is handed out, its error against 64 bits is at most that of the arithmetic in which
    items are cut into runs of `run` tiles, P is rounded to bf16 relative to its run's running maximum (the opening
    tile's, re-based for 32 rows together by more than 2^8 only, and looked at again only where a row sum reaches 2^16 or
    the segment ends) and the runs are added in 64 bits."""
    g = torch.Generator(device="cuda").manual_seed(N + nB)
    r = lambda n, s=1.0: (torch.randn(n, N, D, generator=g, device="cuda") * s).to(torch.bfloat16)
    Q, Kc, Vc, Kq, Vq = r(Lq, q_scale), r(nB), r(nB), r(Lq), r(Lq)
    shape = pafu.Shape(N, D, None, [0, Lq])
    ws = torch.zeros(pafu.pafu_workspace_bytes(shape), dtype=torch.uint8, device="cuda")
    O = torch.empty_like(Q)
    pafu.pafu_chunk_attn(Q, Kc, Vc, [0, nB], Kq, Vq, shape, 0.0, O, None, ws)
    assert pafu.pafu_workspace_status(ws) == 0
    edges = list(range(0, nB, 64)) + list(range(nB, nB + Lq, 64)) + [nB + Lq]
    some = lambda x: torch.nn.functional.pad(x, (0, -Lq % 32)).view(-1, 32).any(1).repeat_interleave(32)[:Lq, None]   # x[Lq], by groups of 32 rows
    e_got = e_cut = 0.0
    for n in range(N):
        k, v = torch.cat([Kc[:, n], Kq[:, n]]).double(), torch.cat([Vc[:, n], Vq[:, n]]).double()
        z = Q[:, n].double() @ k.T * (D ** -0.5 / np.log(2.0))
        want = torch.softmax(z * np.log(2.0), 1) @ v
        top, o, l = z.max(1).values[:, None], 0.0, 0.0
        for t0 in range(0, len(edges) - 1, run):
            m, o_run, l_run = None, 0.0, 0.0
            for t in range(t0, min(t0 + run, len(edges) - 1)):
                zt, vt = z[:, edges[t]:edges[t + 1]], v[edges[t]:edges[t + 1]]
                mx = zt.max(1).values[:, None]
                if m is None:
                    m = mx
                else:
                    look = some((torch.exp2(zt - m).sum(1) >= 65536)) if zt.shape[1] == 64 else torch.ones_like(mx, dtype=torch.bool)
                    m_new = torch.where(look & some((mx - m)[:, 0] > 8), torch.maximum(mx, m), m)
                    o_run, l_run, m = o_run * torch.exp2(m - m_new), l_run * torch.exp2(m - m_new), m_new
                p = torch.exp2(zt - m)
                o_run, l_run = o_run + p.to(torch.bfloat16).double() @ vt, l_run + p.sum(1, keepdim=True)
            o, l = o + torch.exp2(m - top) * o_run, l + torch.exp2(m - top) * l_run
        e_got += float(((O[:, n].double() - want) ** 2).sum())
        e_cut += float((((o / l).to(torch.bfloat16).double() - want) ** 2).sum())
    print("error relative to the pieces': %.4f" % (e_got / e_cut) ** 0.5)
    # both are sums over Lq N D independent roundings: their ratio scatters by about (Lq N D / row correlation)^-1/2 < 1 %
    assert e_got <= 1.02 * e_cut


def test_attention_bounded_wait_runs_out_and_recovers():
    """Every wait in the kernels is bounded.  With the workspace header's test hook set, the
    attention kernel's loader issues no copies: the MMA issuers' and softmax warps' waits run out,
    every role leaves its loop, tensor memory is released, the launch ends and the header holds a
    time-out code.  Nothing faults; after the header is cleared the same workspace serves a
    normal call whose result matches the oracle."""
    N, D, Lq, nB = 2, 128, 300, 500
    d = wl.peaked_attention_inputs("scaled_q", N, D, Lq, nB, seed=2, q_scale=1.0)
    dQ, dKc, dVc, dKq, dVq = [to_device_bf16(d[k]) for k in ("Q", "Kc", "Vc", "Kq", "Vq")]
    shape = pafu.Shape(N, D, None, [0, Lq])
    ws = torch.zeros(pafu.pafu_workspace_bytes(shape), dtype=torch.uint8, device="cuda")
    O = torch.zeros((Lq, N, D), dtype=torch.bfloat16, device="cuda"); LSE = torch.zeros((N, Lq), device="cuda")
    ws.view(torch.int32)[32] = 1                                 # the hook: word 32 of the header
    pafu.pafu_chunk_attn(dQ, dKc, dVc, [0, nB], dKq, dVq, shape, 0.0, O, LSE, ws)     # returns: the launch is asynchronous
    assert pafu.pafu_workspace_status(ws) == 7                   # PAFU_ERR_TIMEOUT, after about half a second
    assert int(ws.view(torch.int32)[0].item()) in (201, 206, 301)  # an issuer's or a softmax warp's first wait
    ws[:256] = 0
    pafu.pafu_chunk_attn(dQ, dKc, dVc, [0, nB], dKq, dVq, shape, 0.0, O, LSE, ws)
    assert pafu.pafu_workspace_status(ws) == 0
    want_O, want_lse = oracle.attention(d["Q"], d["Kc"], d["Vc"], d["Kq"], d["Vq"])
    close(wl.bf16_bits_to_f32(bf16_to_bits(O)), want_O, "after time-out O")
    close(LSE.cpu().numpy(), want_lse, "after time-out LSE")


# ------------------------------------------------- one index list for all layers; Algorithm 2
def test_algorithm2_cache_update_over_chunks():
    """Algorithm 2 run chunk by chunk: the S-MLP scores the new chunk's [q, k, v] at the final
    layer, the salience list SL is carried with the cache, and when the cache would overflow the
    Top-k of SL (plus the sink prefix) is kept in EVERY layer's cache with one index list.  A
    numpy mirror is advanced with the oracle's select / compact from the same fp32 scores; the
    caches and SL must stay bit-identical, the scores within tolerance of the oracle's."""
    rng = np.random.default_rng(31)
    N, D, n_layers, chunk, cap, n_sink = 2, 128, 3, 96, 320, 32
    dm = N * D
    bits = lambda shape, sc=1.0: wl.f32_to_bf16_bits((rng.standard_normal(shape) * sc).astype(np.float32))
    w1, b1 = bits((64, 3 * dm), (3 * dm) ** -0.5), bits((64,), 0.3)
    w2, b2 = bits((12, 64), 64 ** -0.5), bits((12,), 0.3)
    dw = [to_device_bf16(a) for a in (w1, b1, w2, b2)]
    head = pafu.Head(dw[0], dw[1], dw[2], dw[3], wl.ACT_SILU, wl.FINAL_NONE)
    ws = torch.zeros(pafu.pafu_workspace_bytes(pafu.Shape(N, D, [0, cap], [0, chunk]), None, head),
                     dtype=torch.uint8, device="cuda")
    K = [np.zeros((0, N, D), np.uint16) for _ in range(n_layers)]; V = [k.copy() for k in K]   # mirror
    SL = np.zeros(0, np.float32)
    dK = [to_device_bf16(k) for k in K]; dV = [to_device_bf16(v) for v in V]
    dSL = torch.zeros(0, device="cuda")
    pruned = 0
    for c in range(7):
        newK = [bits((chunk, N, D)) for _ in range(n_layers)]; newV = [bits((chunk, N, D)) for _ in range(n_layers)]
        if c == 0:
            first_K = newK
        q = bits((chunk, N, D))
        s_new = torch.full((chunk,), float("nan"), device="cuda")
        pafu.pafu_score_qkv(head, to_device_bf16(q), to_device_bf16(newK[-1]), to_device_bf16(newV[-1]), s_new, ws,
                            ld=dm)
        X = np.concatenate([q.reshape(chunk, dm), newK[-1].reshape(chunk, dm), newV[-1].reshape(chunk, dm)], axis=1)
        close(s_new.cpu().numpy(), oracle.score(np.ascontiguousarray(X), w1, b1, w2, b2, wl.ACT_SILU, wl.FINAL_NONE),
              "chunk score")
        T = SL.shape[0]
        if T + chunk > cap:
            budget = cap - chunk
            shape = pafu.Shape(N, D, [0, T], None)
            pol = pafu.make_policy(n_sink, 0, [budget], 1)
            idx = torch.full((budget,), -1, dtype=torch.int32, device="cuda")
            pafu.pafu_select(dSL, shape, pol, idx)
            want_idx = oracle.select(SL, n_sink, 0, budget)
            assert np.array_equal(idx.cpu().numpy(), want_idx)
            Kc = [torch.zeros((budget, N, D), dtype=torch.bfloat16, device="cuda") for _ in range(n_layers)]
            Vc = [torch.zeros_like(k) for k in Kc]
            SLc = torch.zeros(budget, device="cuda")
            pafu.pafu_compact_layers(dK, dV, dSL, idx, shape, pol, Kc, Vc, SLc)
            K = [oracle.compact(k, want_idx) for k in K]; V = [oracle.compact(v, want_idx) for v in V]
            SL = oracle.compact(SL, want_idx)
            dK, dV, dSL = Kc, Vc, SLc
            pruned += 1
        # append the new chunk (its scores are the GPU's own fp32 values on both sides)
        s_host = s_new.cpu().numpy()
        K = [np.concatenate([a, b]) for a, b in zip(K, newK)]; V = [np.concatenate([a, b]) for a, b in zip(V, newV)]
        SL = np.concatenate([SL, s_host])
        dK = [torch.cat([a, to_device_bf16(b)]) for a, b in zip(dK, newK)]
        dV = [torch.cat([a, to_device_bf16(b)]) for a, b in zip(dV, newV)]
        dSL = torch.cat([dSL, s_new])
        assert SL.shape[0] <= cap
        for l in range(n_layers):
            assert np.array_equal(bf16_to_bits(dK[l]), K[l]) and np.array_equal(bf16_to_bits(dV[l]), V[l]), (c, l)
        assert np.array_equal(dSL.cpu().numpy(), SL)
    # the sink prefix (first tokens of the first chunk) survives every pruning round in every layer
    assert pruned >= 3
    for l in range(n_layers):
        assert np.array_equal(K[l][:n_sink], first_K[l][:n_sink])


@pytest.mark.parametrize("chunk,cap,n_sink", [(96, 320, 32), (101, 323, 17), (64, 64, 8)])
def test_cache_update_entry_point_over_chunks(chunk, cap, n_sink):
    """pafu_cache_update (Algorithm 2's whole per-chunk update in one call: prune every layer with
    one index list when the chunk does not fit, score the chunk into the tail of SL, append the
    chunk's rows) against oracle.cache_update, chunk after chunk: caches, SL and the index list
    bit-identical (the mirror appends the GPU's own fp32 scores), the scores within tolerance of
    the oracle's S-MLP.  Sizes with a ragged tail, an SL tail that is not 16-byte aligned, and a
    cache that holds exactly one chunk (every update replaces everything)."""
    rng = np.random.default_rng(41)
    N, D, n_layers = 2, 128, 3
    dm = N * D
    bits = lambda shape, sc=1.0: wl.f32_to_bf16_bits((rng.standard_normal(shape) * sc).astype(np.float32))
    w1, b1 = bits((64, 3 * dm), (3 * dm) ** -0.5), bits((64,), 0.3)
    w2, b2 = bits((12, 64), 64 ** -0.5), bits((12,), 0.3)
    dw = [to_device_bf16(a) for a in (w1, b1, w2, b2)]
    head = pafu.Head(dw[0], dw[1], dw[2], dw[3], wl.ACT_SILU, wl.FINAL_NONE)
    ws = torch.zeros(pafu.pafu_workspace_bytes(pafu.Shape(N, D, [0, cap], [0, chunk]), None, head),
                     dtype=torch.uint8, device="cuda")
    cache = pafu.Cache(n_layers, N, D, cap, n_sink)
    K = [np.zeros((0, N, D), np.uint16) for _ in range(n_layers)]; V = [k.copy() for k in K]     # mirror
    SL = np.zeros(0, np.float32)
    n_pruned = 0
    for c in range(7):
        newK = [bits((chunk, N, D)) for _ in range(n_layers)]; newV = [bits((chunk, N, D)) for _ in range(n_layers)]
        q = bits((chunk, N, D))
        T_before, cur_before = cache.T, cache.cur
        pruned = pafu.pafu_cache_update(cache, head, to_device_bf16(q), to_device_bf16(newK[-1]), to_device_bf16(newV[-1]),
                                        [to_device_bf16(a) for a in newK], [to_device_bf16(a) for a in newV], ws)
        assert pruned == (T_before + chunk > cap) and cache.cur == (cur_before ^ int(pruned))
        n_pruned += int(pruned)
        assert pafu.pafu_workspace_status(ws) == 0
        s_gpu = cache.SL[cache.T - chunk:].cpu().numpy()
        X = np.concatenate([q.reshape(chunk, dm), newK[-1].reshape(chunk, dm), newV[-1].reshape(chunk, dm)], axis=1)
        close(s_gpu, oracle.score(np.ascontiguousarray(X), w1, b1, w2, b2, wl.ACT_SILU, wl.FINAL_NONE), "chunk score")
        K, V, SL, ids = oracle.cache_update(K, V, SL, newK, newV, s_gpu, cap, n_sink)
        assert (ids is not None) == pruned
        if pruned:
            assert np.array_equal(cache.idx[: cap - chunk].cpu().numpy(), ids)
        assert cache.T == SL.shape[0] <= cap
        assert np.array_equal(cache.SL.cpu().numpy(), SL)
        for l in range(n_layers):
            assert np.array_equal(bf16_to_bits(cache.K[l]), K[l]) and np.array_equal(bf16_to_bits(cache.V[l]), V[l]), (c, l)
    assert n_pruned >= 3


@pytest.mark.parametrize("cap,chunk,N", [
    (1000, 200, 1),                # one selecting CTA
    (4096 + 16 + 129, 129, 1),     # 129 candidates more than it takes: two
    (9000, 700, 1), (24576 + 16 + 129, 129, 1),    # four, eight
    (60001, 700, 1),               # eight with longer shares
    (24592, 8000, 25), (33100, 8000, 25),          # appends that cover the selection: one CTA with the most it takes there, two
    (363001, 800, 1),              # more candidates than a cluster holds: the streaming selection
    # rows of 8, 24, 56 and 200 sixteen-byte units: the 192-unit batches of the row copies hold whole rows, end inside
    # one, or are shorter than one; one row kept or new
    (97, 96, 1), (131, 1, 3), (700, 333, 7), (777, 100, 25), (24, 23, 25), (1500, 1, 7),
])
def test_cache_updates_without_a_synchronisation_between_them(cap, chunk, N):
    """Three updates of a full cache enqueued back to back: each one's selection, copies and head overlap, and the
    next one starts behind them.  Against the oracle's selection on the scores the head gives for the same rows."""
    D, n_layers, n_sink = 64, 2, 16
    g = torch.Generator(device="cuda").manual_seed(cap)
    rows = lambda n: torch.randn(n, N, D, generator=g, device="cuda").to(torch.bfloat16)
    w = [torch.randn(*s, generator=g, device="cuda").to(torch.bfloat16) / 8 for s in ((64, 3 * N * D), (64,), (12, 64), (12,))]
    head = pafu.Head(*w, wl.ACT_SILU, wl.FINAL_NONE)
    ws = torch.zeros(pafu.pafu_workspace_bytes(pafu.Shape(N, D, [0, cap], [0, chunk]), None, head), dtype=torch.uint8, device="cuda")
    cache = pafu.Cache(n_layers, N, D, cap, n_sink)
    K, V = [rows(cap) for _ in range(n_layers)], [rows(cap) for _ in range(n_layers)]
    for l in range(n_layers):
        cache.Kb[0][l].copy_(K[l]); cache.Vb[0][l].copy_(V[l])
    SL = torch.randn(cap, generator=g, device="cuda")
    cache.SLb[0].copy_(SL)
    cache.c.T = cap
    chunks = [(rows(chunk), [rows(chunk) for _ in range(n_layers)], [rows(chunk) for _ in range(n_layers)]) for _ in range(3)]
    torch.cuda.synchronize()
    for q, kn, vn in chunks:
        assert pafu.pafu_cache_update(cache, head, q, kn[-1], vn[-1], kn, vn, ws)
    assert pafu.pafu_workspace_status(ws) == 0
    for q, kn, vn in chunks:
        ids = oracle.select(SL.cpu().numpy(), n_sink, 0, cap - chunk)
        i = torch.from_numpy(ids.astype(np.int64)).cuda()
        s = torch.empty(chunk, device="cuda")
        pafu.pafu_score_qkv(head, q, kn[-1], vn[-1], s, ws, ld=N * D)
        K = [torch.cat([a[i], b]) for a, b in zip(K, kn)]; V = [torch.cat([a[i], b]) for a, b in zip(V, vn)]
        SL = torch.cat([SL[i], s])
    assert np.array_equal(cache.idx[: cap - chunk].cpu().numpy(), ids)
    assert torch.equal(cache.SL, SL)
    for l in range(n_layers):
        assert torch.equal(cache.K[l], K[l]) and torch.equal(cache.V[l], V[l])


@pytest.mark.parametrize("layers,N,cap,chunk,hidden", [
    (1, 8, 700, 130, 1024),       # short copies: the head shares their SMs, (tile, chunk) units in clusters of four
    (3, 4, 2000, 1900, 640),      # the same with a half-full last accumulator
    (2, 4, 1000, 700, 64),        # one accumulator: tiles shared by two CTAs
    (40, 4, 3000, 300, 256),      # copies too long for that
    (4, 2, 1000, 500, 1024),      # too narrow a head for that
    (3, 12, 4000, 128, 16),       # one CTA on the SM that selects
    (3, 12, 12000, 130, 64), (2, 12, 12000, 128, 1024),    # four on those of a selecting cluster
    (3, 12, 12000, 257, 64),      # more than those
])
def test_cache_update_head_beside_the_copies(layers, N, cap, chunk, hidden):
    """The salience head beside the row copies, on their SMs or not, gives the bits that it gives alone; the rows are copies."""
    D, keep = 128, cap - chunk
    g = torch.Generator(device="cuda").manual_seed(layers + hidden)
    rn = lambda *shape: torch.randn(*shape, generator=g, device="cuda")
    w = [(rn(*s) / 8).to(torch.bfloat16) for s in ((hidden, 3 * N * D), (hidden,), (12, hidden), (12,))]
    head = pafu.Head(*w, wl.ACT_SILU, wl.FINAL_NONE)
    ws = torch.zeros(pafu.pafu_workspace_bytes(pafu.Shape(N, D, [0, cap], [0, chunk]), None, head), dtype=torch.uint8, device="cuda")
    cache = pafu.Cache(layers, N, D, cap, 50)
    for l in range(layers):
        cache.Kb[0][l].copy_(rn(cap, N, D)); cache.Vb[0][l].copy_(rn(cap, N, D))
    cache.SLb[0].copy_(rn(cap))
    cache.c.T = cap
    new = [rn(chunk, N, D).to(torch.bfloat16) for _ in range(3)]
    want = torch.empty(chunk, device="cuda")
    pafu.pafu_score_qkv(head, *new, want, ws, ld=N * D)
    for _ in range(3):                                     # back to back from the same full cache
        cache.c.T, cache.c.cur = cap, 0
        pafu.pafu_cache_update(cache, head, *new, [new[1]] * layers, [new[2]] * layers, ws)
    assert pafu.pafu_workspace_status(ws) == 0
    assert torch.equal(cache.SL[keep:], want)
    i = cache.idx[:keep].long()
    assert torch.equal(cache.SL[:keep], cache.SLb[0][:cap][i])
    for l in range(layers):
        assert torch.equal(cache.K[l], torch.cat([cache.Kb[0][l][i], new[1]]))
        assert torch.equal(cache.V[l], torch.cat([cache.Vb[0][l][i], new[2]]))


@pytest.mark.parametrize("T,where", [(300, "append"), (128, "append"), (300, "kept"), (256, "append")])
def test_cache_update_head_inputs_in_the_idle_buffers(T, where):
    """The head's input rows may lie in buffers that the update writes: in rows that the append overwrites (they are
    read before), or in rows that the gather fills (they are read after).  Pruning (T = 300, 256), nothing kept (a chunk of the
    whole capacity at T = 256) and not pruning (T = 128)."""
    N, D, n_layers, cap = 2, 128, 3, 300
    chunk = cap if T == 256 else 150
    rng = np.random.default_rng(T)
    rows = lambda n: to_device_bf16(wl.f32_to_bf16_bits(rng.standard_normal((n, N, D)).astype(np.float32)))
    w1, w2 = rng.standard_normal((64, 3 * N * D)) / 30, rng.standard_normal((12, 64)) / 8
    head = pafu.Head(*[to_device_bf16(wl.f32_to_bf16_bits(w.astype(np.float32))) for w in (w1, w1[:, 0], w2, w2[:, 0])],
                     wl.ACT_SILU, wl.FINAL_NONE)
    ws = torch.zeros(pafu.pafu_workspace_bytes(pafu.Shape(N, D, [0, cap], [0, chunk]), None, head), dtype=torch.uint8, device="cuda")
    old = [[rows(cap) for _ in range(n_layers)] for _ in range(2)]
    new = [[rows(chunk) for _ in range(n_layers)] for _ in range(2)]
    SL, q = torch.randn(cap, generator=torch.Generator().manual_seed(T)), rows(chunk)
    res = []
    for inside in (False, True):
        cache = pafu.Cache(n_layers, N, D, cap, 16)
        for l in range(n_layers):
            cache.Kb[0][l].copy_(old[0][l]); cache.Vb[0][l].copy_(old[1][l])
        cache.SLb[0].copy_(SL)
        cache.c.T = T
        prune = T + chunk > cap
        to, dst = (1, cap - chunk) if prune else (0, T)
        Qs, Ks, Vs = q, new[0][-1], new[1][-1]
        if where == "kept":                               # the first `chunk` rows that the pruning keeps in layer 1
            kept = np.sort(np.concatenate([np.arange(16), 16 + np.argsort(-SL.numpy()[16:T], kind="stable")[: cap - chunk - 16]]))
            Qs = old[0][1][torch.from_numpy(kept).cuda()]
            if inside:
                Qs = cache.Kb[to][1][:chunk]
        elif inside:
            cache.Kb[to][0][dst:dst + chunk].copy_(q); Qs = cache.Kb[to][0][dst:dst + chunk]
            cache.Vb[to][2][dst:dst + chunk].copy_(Vs); Vs = cache.Vb[to][2][dst:dst + chunk]
        assert pafu.pafu_cache_update(cache, head, Qs, Ks, Vs, new[0], new[1], ws) == prune
        assert pafu.pafu_workspace_status(ws) == 0
        res.append([t.clone() for t in [cache.SL] + cache.K + cache.V])
    for a, b in zip(*res):
        assert torch.equal(a, b)


# --------------------------------------------------------------- attention through indices
def test_indexed_attention_matches_oracle_and_compacted_path():
    """Select(KV; ids) applied inside the attention loader (Eq. 7's index set) instead of as a
    copy: against the oracle on the oracle's own gathered rows, and bit-equal to the CUDA path
    that compacts first.  Retained counts sit around the 4-row gather and 64-key tile sizes;
    streams have non-zero offsets into the packed cache."""
    rng = np.random.default_rng(21)
    N, D = 3, 128
    for T, Bs, Lq, chunk in [((300,), (1,), (5,), False), ((300,), (3,), (70,), True),
                             ((500, 129, 1000), (63, 129, 257), (130, 1, 300), True),
                             ((257, 64), (65, 64), (256, 257), False),
                             ((2000,), (1027,), (520,), True)]:
        n = len(T)
        cuT = np.concatenate([[0], np.cumsum(T)]); cuB = np.concatenate([[0], np.cumsum(Bs)])
        cuQ = np.concatenate([[0], np.cumsum(Lq)])
        bits = lambda m: wl.f32_to_bf16_bits(rng.standard_normal((m, N, D)).astype(np.float32))
        K, V, Q, Kq, Vq = bits(cuT[-1]), bits(cuT[-1]), bits(cuQ[-1]), bits(cuQ[-1]), bits(cuQ[-1])
        idx = np.concatenate([np.sort(rng.choice(T[s], size=Bs[s], replace=False)) for s in range(n)]).astype(np.int32)
        shape = pafu.Shape(N, D, cuT, cuQ)
        pol = pafu.make_policy(0, 0, list(Bs), n)
        dK, dV, dQ, dKq, dVq = [to_device_bf16(a) for a in (K, V, Q, Kq, Vq)]
        didx = torch.from_numpy(idx).cuda()
        ws = torch.zeros(pafu.pafu_workspace_bytes(shape), dtype=torch.uint8, device="cuda")
        O = torch.full((int(cuQ[-1]), N, D), float("nan"), dtype=torch.bfloat16, device="cuda")
        LSE = torch.full((N, int(cuQ[-1])), float("nan"), device="cuda")
        pafu.pafu_chunk_attn_indexed(dQ, dK, dV, didx, cuB, dKq if chunk else None, dVq if chunk else None,
                                     shape, 0.0, O, LSE, ws)
        assert pafu.pafu_workspace_status(ws) == 0
        got = wl.bf16_bits_to_f32(bf16_to_bits(O)); lse = LSE.cpu().numpy()
        for s in range(n):
            i = idx[cuB[s]:cuB[s + 1]]
            want, wlse = oracle.attention(Q[cuQ[s]:cuQ[s + 1]], oracle.compact(K[cuT[s]:cuT[s + 1]], i),
                                          oracle.compact(V[cuT[s]:cuT[s + 1]], i),
                                          Kq[cuQ[s]:cuQ[s + 1]] if chunk else None,
                                          Vq[cuQ[s]:cuQ[s + 1]] if chunk else None)
            close(got[cuQ[s]:cuQ[s + 1]], want, "indexed O %s stream %d" % ((T, Bs, Lq), s))
            close(lse[:, cuQ[s]:cuQ[s + 1]], wlse, "indexed LSE")
        # the compact-then-attend path on the same inputs gives the same bits
        Kc = torch.zeros((int(cuB[-1]), N, D), dtype=torch.bfloat16, device="cuda"); Vc = torch.zeros_like(Kc)
        pafu.pafu_compact(dK, dV, None, didx, shape, pol, Kc, Vc, None)
        O2 = torch.full_like(O, float("nan")); LSE2 = torch.full_like(LSE, float("nan"))
        pafu.pafu_chunk_attn(dQ, Kc, Vc, cuB, dKq if chunk else None, dVq if chunk else None, shape, 0.0, O2, LSE2, ws)
        assert torch.equal(O.view(torch.int16), O2.view(torch.int16)) and torch.equal(LSE, LSE2)


@pytest.mark.parametrize("w", [wl.small_ragged(2, 128), wl.wan13b_layer(), wl.wan13b_layer(0.25), wl.paper_native(),
                               wl.long_horizon(), wl.batch4_14b()],
                         ids=lambda w: "%s-B%d" % (w.name, w.budget[0]))
def test_step_indexed_equals_step(w):
    d = wl.make_layer(w)
    A = Layer(w, d); B = Layer(w, d)
    A.step(); A.check_status()
    B.O.fill_(float("nan")); B.LSE.fill_(float("nan"))
    B.step_indexed(); B.check_status()
    assert torch.equal(A.scores[: A.nT], B.scores[: A.nT])
    assert torch.equal(A.idx[: A.nB], B.idx[: A.nB])
    assert torch.equal(A.O.view(torch.int16), B.O.view(torch.int16))
    assert torch.equal(A.LSE, B.LSE)


@pytest.mark.parametrize("N,D,Lq,nB", [
    (1, 128, 1, 1), (2, 64, 64, 128),                         # whole items, one round, nothing to merge
    (3, 128, 129, 500),                                       # 11 tiles an item, one tile a CTA: 11 pieces
    (1, 128, 130, 64 * 40 + 1), (1, 64, 300, 64 * 40 - 1),    # one or two items over many CTAs: about 40 pieces
    (2, 128, 257, 64 * 20 + 5),                               # a one-row tail item; over 20 pieces
    (3, 128, 2000, 64 * 9),                                   # seven pieces: the merge for few pieces
    (40, 128, 1100, 100),                                     # more items than CTAs: a whole round, then shares
    (6, 64, 1900, 700), (30, 64, 515, 900),                   # d_head 64: two to four pieces, a three-row tail item
])
def test_attention_work_split(N, D, Lq, nB):
    """The ways a problem is handed to the CTAs (whole items, shares, a round of whole items followed by shares) and
    the merges they lead to."""
    d = wl.peaked_attention_inputs("scaled_q", N, D, Lq, nB, seed=Lq, q_scale=2.0)
    shape = pafu.Shape(N, D, None, [0, Lq])
    ws = torch.zeros(pafu.pafu_workspace_bytes(shape), dtype=torch.uint8, device="cuda")
    O = torch.full((Lq, N, D), float("nan"), dtype=torch.bfloat16, device="cuda")
    LSE = torch.full((N, Lq), float("nan"), device="cuda")
    t = {k: to_device_bf16(v) for k, v in d.items()}
    pafu.pafu_chunk_attn(t["Q"], t["Kc"], t["Vc"], [0, nB], t["Kq"], t["Vq"], shape, 0.0, O, LSE, ws)
    assert pafu.pafu_workspace_status(ws) == 0
    want, want_lse = oracle.attention(d["Q"], d["Kc"], d["Vc"], d["Kq"], d["Vq"])
    close(O.float().cpu().numpy(), want, "O", scaled=True)
    # 32-bit sums and logits of a few tens: 1e-5 is ten units in the last place
    np.testing.assert_allclose(LSE.cpu().numpy(), want_lse, rtol=1e-5, atol=1e-5)


@pytest.mark.parametrize("nB", [2, 64 * 300])                  # one CTA; merged from the pieces of many
@pytest.mark.parametrize("D", [64, 128])
def test_lse_is_rounded_once(D, nB):
    """LSE = m scale + log l is one fused operation: nB equal keys and integer logits give exact maxima and sums, so the
    result is off by its own rounding (half a unit) and logf's (at most one unit of log l), and not by a rounding of m scale as
    well.  The scale is one whose product with log2 e is exactly 1/8, so that every probability is 1."""
    Lq, N = 300, 2
    log2e = np.float32(1.4426950408889634)
    s0 = np.float32(0.125 / 1.4426950408889634)
    scale = next(s for s in (s0, np.nextafter(s0, np.float32(1)), np.nextafter(s0, np.float32(0))) if s * log2e == np.float32(0.125))
    rng = np.random.default_rng(D + nB)
    q = rng.integers(0, 200, (Lq, N, D)).astype(np.float32)     # at most 8 bits: exact in bf16, dot products exact in 32 bits
    Q = to_device_bf16(wl.f32_to_bf16_bits(q))
    K = torch.ones((nB, N, D), dtype=torch.bfloat16, device="cuda")
    shape = pafu.Shape(N, D, None, [0, Lq])
    ws = torch.zeros(pafu.pafu_workspace_bytes(shape), dtype=torch.uint8, device="cuda")
    O, LSE = torch.empty_like(Q), torch.empty((N, Lq), device="cuda")
    pafu.pafu_chunk_attn(Q, K, K, [0, nB], None, None, shape, float(scale), O, LSE, ws)
    assert pafu.pafu_workspace_status(ws) == 0
    want = q.sum(2).T.astype(np.float64) * float(scale) + np.log(float(nB))
    bound = 0.5 * np.spacing(want.astype(np.float32)).astype(np.float64) * 1.0001 + np.spacing(np.float32(np.log(nB)))
    err = np.abs(LSE.cpu().numpy().astype(np.float64) - want)
    assert np.all(err <= bound), (err / bound).max()


# ------------------------------------------------------------- teacher salience (Eq. 4, Eq. 5)
@pytest.mark.parametrize("L,N,LB", [
    (700, 2, 200),      # four blocks, the last one half length; every tile ragged
    (1024, 3, 256),     # blocks that are whole tiles
    (300, 1, 300),      # a single block
    (130, 2, 64),       # blocks smaller than a tile
    (3 * 1560, 2, 1560),  # three frames as blocks: several tiles and key-tile pairs per block
])
def test_sse_matches_oracle(L, N, LB):
    rng = np.random.default_rng(L + N)
    D = 128
    # logits with a few dominant keys per row, as attention maps have
    Q = wl.f32_to_bf16_bits((rng.standard_normal((L, N, D)) * 1.5).astype(np.float32))
    K = wl.f32_to_bf16_bits((rng.standard_normal((L, N, D)) * 1.5).astype(np.float32))
    want_s, want_c = oracle.sse(Q, K, LB)
    dQ, dK = to_device_bf16(Q), to_device_bf16(K)
    ws = torch.zeros(pafu.pafu_sse_workspace_bytes(L, N, D, LB), dtype=torch.uint8, device="cuda")
    s = torch.full((L,), float("nan"), device="cuda"); comp = torch.full((3, L), float("nan"), device="cuda")
    gmax = torch.full((L,), float("nan"), device="cuda")
    gavg = torch.full((L,), float("nan"), device="cuda")
    pafu.pafu_sse(dQ, dK, None, LB, 0.0, s, comp, ws, gmax=gmax, gavg=gavg)
    assert pafu.pafu_workspace_status(ws) == 0
    tol = dict(rtol=1e-3, atol=1e-7)
    assert np.allclose(gmax.cpu().numpy(), oracle.sse_global_max(Q, K), **tol)    # the "Max" ablation
    assert np.allclose(gavg.cpu().numpy(), oracle.sse_global_avg(Q, K), **tol)    # the "Avg" ablation
    assert np.allclose(comp.cpu().numpy(), want_c, **tol), np.abs(comp.cpu().numpy() - want_c).max()
    assert np.allclose(s.cpu().numpy(), want_s, **tol)
    # with the row statistics handed in (as the attention call leaves them) the result is the same
    shape = pafu.Shape(N, D, None, [0, L])
    ws2 = torch.zeros(pafu.pafu_workspace_bytes(shape), dtype=torch.uint8, device="cuda")
    O = torch.empty((L, N, D), dtype=torch.bfloat16, device="cuda"); LSE = torch.empty((N, L), device="cuda")
    pafu.pafu_chunk_attn(dQ, dK, dK, [0, L], None, None, shape, 0.0, O, LSE, ws2)
    s2 = torch.full_like(s, float("nan"))
    pafu.pafu_sse(dQ, dK, LSE, LB, 0.0, s2, None, ws)
    assert pafu.pafu_workspace_status(ws) == 0
    assert torch.equal(s, s2)


@pytest.mark.parametrize("rise", [0.0, 4.0, -4.0, 20.0, -20.0])
@pytest.mark.parametrize("L,N", [(1, 2), (64, 2), (65, 2), (128, 2), (129, 2), (256, 2), (257, 2), (640, 2), (1100, 2),   # runs of one to four tiles
                                 (4000, 2),      # runs of 13 tiles: past the nine K stages and the four S buffers
                                 (1100, 40)])    # whole items of 18 tiles and shares of what is left
def test_sse_row_statistics(L, N, rise):
    """The pass that computes the row log-sum-exps (LSE = NULL): sequence lengths around its 64-token key tiles, pairs of
    128-row query tiles and rings of buffers, and logits that rise or fall by `rise` nats per 64 keys: in a run of
    several tiles the opening tile's maximum then goes stale, is outgrown beyond a row sum of 2^16 again and again,
    or holds for good.  The same bits as with the log-sum-exps of the attention kernel."""
    D, LB = 128, max(1, L // 3)
    rng = np.random.default_rng(L)
    Q = rng.standard_normal((L, N, D), dtype=np.float32) + 1.0
    K = rng.standard_normal((L, N, D), dtype=np.float32) + (rise / np.sqrt(D) * np.arange(L, dtype=np.float32) / 64)[:, None, None]
    Q, K = wl.f32_to_bf16_bits(Q), wl.f32_to_bf16_bits(K.astype(np.float32))
    want, _ = oracle.sse(Q, K, LB)
    s = torch.empty(L, dtype=torch.float32, device="cuda")
    ws = torch.zeros(pafu.pafu_sse_workspace_bytes(L, N, D, LB), dtype=torch.uint8, device="cuda")
    pafu.pafu_sse(to_device_bf16(Q), to_device_bf16(K), None, LB, 0.0, s, None, ws)
    assert pafu.pafu_workspace_status(ws) == 0
    # s = exp(z - lse): 32-bit logits and sums of magnitude up to max|z| lose a few units of 2^-24 max|z|
    zmax = 1.0 + np.abs(wl.bf16_bits_to_f32(Q).reshape(L, -1)).sum(1).max() * np.abs(wl.bf16_bits_to_f32(K)).max() / np.sqrt(D)
    np.testing.assert_allclose(s.cpu().numpy(), want, rtol=8 * 2.0 ** -24 * zmax + 1e-6, atol=1e-30)
    q, k = to_device_bf16(Q), to_device_bf16(K)
    shape = pafu.Shape(N, D, None, [0, L])
    ws2 = torch.zeros(pafu.pafu_workspace_bytes(shape), dtype=torch.uint8, device="cuda")
    LSE, s2 = torch.empty((N, L), device="cuda"), torch.empty_like(s)
    pafu.pafu_chunk_attn(q, k, k, [0, L], None, None, shape, 0.0, torch.empty_like(q), LSE, ws2)
    pafu.pafu_sse(q, k, LSE, LB, 0.0, s2, None, ws)
    assert torch.equal(s, s2)
    if L == 4000 and rise == 20.0:
        c = pafu.pafu_workspace_counters(ws2)
        assert c[1] > 0 and c[2] > 0      # such an input does send tiles through the redo and the re-base


def test_sse_row_statistics_bounded_wait_runs_out_and_recovers():
    """The row-statistics pass with its loader stalled (the header's test hook): every role's wait runs out, the launch
    ends, the header holds a time-out code of that pass, and after it is cleared the workspace serves a normal call."""
    L, N, D, LB = 700, 2, 128, 200
    rng = np.random.default_rng(4)
    Q, K = [wl.f32_to_bf16_bits(rng.standard_normal((L, N, D), dtype=np.float32)) for _ in range(2)]
    q, k, s = to_device_bf16(Q), to_device_bf16(K), torch.zeros(L, device="cuda")
    ws = torch.zeros(pafu.pafu_sse_workspace_bytes(L, N, D, LB), dtype=torch.uint8, device="cuda")
    ws.view(torch.int32)[32] = 1
    pafu.pafu_sse(q, k, None, LB, 0.0, s, None, ws)
    assert pafu.pafu_workspace_status(ws) == 7                   # PAFU_ERR_TIMEOUT, after about half a second
    assert int(ws.view(torch.int32)[0].item()) in (711, 712, 721)
    ws[:256] = 0
    pafu.pafu_sse(q, k, None, LB, 0.0, s, None, ws)
    assert pafu.pafu_workspace_status(ws) == 0
    want, _ = oracle.sse(Q, K, LB)
    np.testing.assert_allclose(s.cpu().numpy(), want, rtol=1e-4, atol=1e-30)   # logits below 100: 8 x 2^-24 x 100 < 1e-4


@pytest.mark.parametrize("L,N,LB", [
    (700, 3, 200),      # four blocks, the last one half length; blocks and 64-token tiles do not line up
    (1024, 2, 256),     # blocks that are whole tiles
    (130, 1, 64),       # one head: Algorithm 3's order and Eq. 4's coincide
])
def test_sse_mean_first_matches_oracle(L, N, LB):
    """Algorithm 3's order of operations (mean over heads, then the maximum over queries) against
    its oracle; with one head also against pafu_sse itself."""
    rng = np.random.default_rng(L * 7 + N)
    D = 128
    Q = wl.f32_to_bf16_bits((rng.standard_normal((L, N, D)) * 1.5).astype(np.float32))
    K = wl.f32_to_bf16_bits((rng.standard_normal((L, N, D)) * 1.5).astype(np.float32))
    want_s, want_c = oracle.sse_mean_first(Q, K, LB)
    dQ, dK = to_device_bf16(Q), to_device_bf16(K)
    ws = torch.zeros(pafu.pafu_sse_workspace_bytes(L, N, D, LB), dtype=torch.uint8, device="cuda")
    s = torch.full((L,), float("nan"), device="cuda"); comp = torch.full((3, L), float("nan"), device="cuda")
    pafu.pafu_sse_mean_first(dQ, dK, None, LB, 0.0, s, comp, ws)
    assert pafu.pafu_workspace_status(ws) == 0
    tol = dict(rtol=1e-3, atol=1e-7)
    assert np.allclose(comp.cpu().numpy(), want_c, **tol), np.abs(comp.cpu().numpy() - want_c).max()
    assert np.allclose(s.cpu().numpy(), want_s, **tol)
    s4 = torch.full_like(s, float("nan")); comp4 = torch.full_like(comp, float("nan"))
    pafu.pafu_sse(dQ, dK, None, LB, 0.0, s4, comp4, ws)
    if N == 1:
        assert np.allclose(comp.cpu().numpy(), comp4.cpu().numpy(), **tol)
    else:
        assert torch.all(comp <= comp4 * (1 + 1e-3) + 1e-7)       # max of the mean <= mean of the maxima


def test_sse_full_size_sampled_columns():
    """The paper's training length (21 frames x 1560 tokens, blocks of 4680; Appendix A), one head:
    a seeded sample of key positions, block and tile boundaries included, against the oracle."""
    L, N, D, LB = 32760, 1, 128, 4680
    rng = np.random.default_rng(3)
    Q = wl.f32_to_bf16_bits((rng.standard_normal((L, N, D)) * 1.5).astype(np.float32))
    K = wl.f32_to_bf16_bits((rng.standard_normal((L, N, D)) * 1.5).astype(np.float32))
    cols = sorted(set([0, 127, 128, LB - 1, LB, LB + 1, 4607, 4608, 2 * LB - 1, 2 * LB, L - LB - 1, L - LB, L - 1])
                  | set(rng.choice(L, size=19, replace=False).tolist()))
    want_s, want_c = oracle.sse_cols(Q, K, LB, cols)
    ws = torch.zeros(pafu.pafu_sse_workspace_bytes(L, N, D, LB), dtype=torch.uint8, device="cuda")
    s = torch.full((L,), float("nan"), device="cuda"); comp = torch.full((3, L), float("nan"), device="cuda")
    pafu.pafu_sse(to_device_bf16(Q), to_device_bf16(K), None, LB, 0.0, s, comp, ws)
    assert pafu.pafu_workspace_status(ws) == 0
    got_s, got_c = s.cpu().numpy(), comp.cpu().numpy()
    assert np.all(np.isfinite(got_s)) and np.all(got_c >= 0) and np.all(got_c <= 1.0 + 1e-5)
    assert np.all(got_c[2, :LB] == 0) and np.all(got_c[0, L - LB:] == 0)     # classes without queries
    assert np.allclose(got_c[:, cols], want_c, rtol=1e-3, atol=1e-7), np.abs(got_c[:, cols] - want_c).max()
    assert np.allclose(got_s[cols], want_s, rtol=1e-3, atol=1e-7)


# ---------------------------------------------------------------------------------- step
@pytest.mark.parametrize("w", SMALL, ids=lambda w: "%s-d%d" % (w.name, w.d_head))
def test_step_equals_four_calls_and_oracle(w):
    d = wl.make_layer(w)
    A = Layer(w, d); B = Layer(w, d)
    A.step(); A.check_status()
    B.score(); B.select(); B.compact(); B.attn(); B.check_status()
    for name in ("scores", "idx", "Kc", "Vc", "SLc", "O", "LSE"):
        a, b = getattr(A, name), getattr(B, name)
        n = {"scores": A.nT, "idx": A.nB, "Kc": A.nB, "Vc": A.nB, "SLc": A.nB}.get(name)
        if n is not None:
            a, b = a[:n], b[:n]
        assert torch.equal(a.view(torch.int16) if a.dtype == torch.bfloat16 else a,
                           b.view(torch.int16) if b.dtype == torch.bfloat16 else b), name
    # against the oracle: scores within tolerance; indices exact given the GPU's own fp32 scores;
    # compacted K/V/SL byte-identical given those indices; attention within tolerance
    gs = A.scores[: A.nT].cpu().numpy()
    close(gs, oracle_scores(w, d), "step scores")
    idx = oracle_select_streams(gs, w)
    got_idx = A.idx[: A.nB].cpu().numpy()
    cuT, cuB, cuQ = w.cu("T"), A.cu_B, w.cu("Lq")
    Kc_bits, Vc_bits = bf16_to_bits(A.Kc)[: A.nB], bf16_to_bits(A.Vc)[: A.nB]
    for s in range(w.n_streams):
        assert np.array_equal(got_idx[cuB[s]:cuB[s + 1]], idx[s])
        assert np.array_equal(Kc_bits[cuB[s]:cuB[s + 1]], oracle.compact(d["K"][cuT[s]:cuT[s + 1]], idx[s]))
        assert np.array_equal(Vc_bits[cuB[s]:cuB[s + 1]], oracle.compact(d["V"][cuT[s]:cuT[s + 1]], idx[s]))
        assert np.array_equal(A.SLc.cpu().numpy()[cuB[s]:cuB[s + 1]], gs[cuT[s]:cuT[s + 1]][idx[s]])
    got = wl.bf16_bits_to_f32(bf16_to_bits(A.O))
    for s, (O, Ls) in enumerate(oracle_attn_streams(w, d, Kc_bits, Vc_bits, cuB)):
        close(got[cuQ[s]:cuQ[s + 1]], O, "step O")


def test_step_host_matches_device_step():
    w = wl.small_ragged(2, 128)
    d = wl.make_layer(w)
    A = Layer(w, d)
    A.step(); A.check_status()
    host = {k: torch.from_numpy(v.view(np.int16)).pin_memory() for k, v in d.items()}
    scores = torch.empty(A.nT, dtype=torch.float32).pin_memory()
    idx = torch.empty(A.nB, dtype=torch.int32).pin_memory()
    O = torch.empty((A.nQ, w.n_heads, w.d_head), dtype=torch.int16).pin_memory()
    head = pafu.Head(host["w1"], host["b1"], host["w2"], host["b2"], w.act, w.final)
    arena = torch.empty(pafu.pafu_step_host_arena_bytes(A.shape, A.policy, head), dtype=torch.uint8, device="cuda")
    args = pafu.step_args(A.shape, head, A.policy, host["K"], host["V"], host["Q"], host["Kq"], host["Vq"],
                          0.0, scores, idx, None, None, None, O, None, None)
    pafu.pafu_step_host(args, arena)
    assert torch.equal(scores, A.scores[: A.nT].cpu())
    assert torch.equal(idx, A.idx[: A.nB].cpu())
    assert torch.equal(O, A.O.view(torch.int16).cpu())


def test_step_host_async_two_steps_in_flight():
    """Two host-buffer steps on two streams with an arena each (the copies of one overlap the
    kernels of the other): after the streams are synchronised both give what the blocking call gives."""
    w = wl.small_ragged(2, 128)
    datas = [wl.make_layer(w, seed=s) for s in (0, 1)]
    want = []
    for d in datas:
        A = Layer(w, d)
        A.step(); A.check_status()
        want.append((A.scores[: A.nT].cpu(), A.idx[: A.nB].cpu(), A.O.view(torch.int16).cpu()))
    shape, policy, nT, nB, nQ = A.shape, A.policy, A.nT, A.nB, A.nQ
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    keep, outs = [], []
    torch.cuda.synchronize()
    for d, st in zip(datas, streams):
        host = {k: torch.from_numpy(v.view(np.int16)).pin_memory() for k, v in d.items()}
        scores = torch.empty(nT, dtype=torch.float32).pin_memory()
        idx = torch.empty(nB, dtype=torch.int32).pin_memory()
        O = torch.empty((nQ, w.n_heads, w.d_head), dtype=torch.int16).pin_memory()
        word = torch.full((1,), -1, dtype=torch.int32).pin_memory()
        head = pafu.Head(host["w1"], host["b1"], host["w2"], host["b2"], w.act, w.final)
        arena = torch.empty(pafu.pafu_step_host_arena_bytes(shape, policy, head), dtype=torch.uint8, device="cuda")
        args = pafu.step_args(shape, head, policy, host["K"], host["V"], host["Q"], host["Kq"], host["Vq"],
                              0.0, scores, idx, None, None, None, O, None, None)
        pafu.pafu_step_host_async(args, arena, word, stream=st)
        keep.append((host, head, arena, args))
        outs.append((scores, idx, O, word))
    for st in streams:
        st.synchronize()
    for (scores, idx, O, word), (ws, wi, wo) in zip(outs, want):
        assert int(word[0]) == 0
        assert torch.equal(scores, ws) and torch.equal(idx, wi) and torch.equal(O, wo)


# ---------------------------------------------------------------------- full-size configs
def _full_size_check(w, n_rows=256, seed=0, score_rows=None, peaked=False):
    d = wl.make_layer(w, seed=seed)
    if peaked:
        # queries that are copies of keys the policy always keeps (sink, recent) or of the chunk's own
        # keys: every row's attention concentrates on a few keys and the outputs are O(1)
        d["Q"] = wl.queries_from_keys(w, d, seed=seed)
    L = Layer(w, d)
    L.step(); L.check_status()
    torch.cuda.synchronize()
    gs = L.scores[: L.nT].cpu().numpy()
    if score_rows is None:
        close(gs, oracle_scores(w, d), "scores")
    else:
        # the oracle's MLP on a seeded sample of tokens (first, last and tile-boundary rows included)
        rows = wl.sample_rows(L.nT, score_rows, seed=seed, tag=77)
        want = oracle.score(d["K"].reshape(L.nT, -1)[rows], d["w1"], d["b1"], d["w2"], d["b2"], w.act, w.final)
        close(gs[rows], want, "scores (sampled)")
    idx = oracle_select_streams(gs, w)
    got_idx = L.idx[: L.nB].cpu().numpy()
    cuT, cuB, cuQ = w.cu("T"), L.cu_B, w.cu("Lq")
    Kc_bits, Vc_bits = bf16_to_bits(L.Kc)[: L.nB], bf16_to_bits(L.Vc)[: L.nB]
    rows = []
    for s in range(w.n_streams):
        assert np.array_equal(got_idx[cuB[s]:cuB[s + 1]], idx[s])
        assert np.array_equal(Kc_bits[cuB[s]:cuB[s + 1]], oracle.compact(d["K"][cuT[s]:cuT[s + 1]], idx[s]))
        assert np.array_equal(Vc_bits[cuB[s]:cuB[s + 1]], oracle.compact(d["V"][cuT[s]:cuT[s + 1]], idx[s]))
        r = set(wl.sample_rows(w.Lq[s], n_rows, seed=seed, tag=s).tolist())
        last_tile = (w.Lq[s] // 128) * 128          # rows of the partial last tile
        r |= set(range(last_tile, w.Lq[s])[:: max(1, (w.Lq[s] - last_tile) // 16)])
        rows.append(np.array(sorted(r), dtype=np.int64))
    got = wl.bf16_bits_to_f32(bf16_to_bits(L.O))
    lse = L.LSE.cpu().numpy()
    for s, (O, Ls) in enumerate(oracle_attn_streams(w, d, Kc_bits, Vc_bits, cuB, rows)):
        close(got[cuQ[s]:cuQ[s + 1]][rows[s]], O, "O stream %d" % s, scaled=peaked)
        close(lse[:, cuQ[s]:cuQ[s + 1]][:, rows[s]], Ls, "LSE stream %d" % s)


def test_full_size_wan13b_layer():
    _full_size_check(wl.wan13b_layer())


def test_full_size_wan13b_layer_peaked_attention():
    _full_size_check(wl.wan13b_layer(), peaked=True, seed=1)


@pytest.mark.parametrize("frac", [0.25, 0.75])
def test_full_size_budget_sweep(frac):
    # the other two budgets of the 30-layer sweep (a different layer's random streams each)
    w = wl.wan13b_layer(frac)
    assert w.budget[0] == {0.25: 7020, 0.75: 21060}[frac]
    _full_size_check(w, n_rows=256, seed=int(frac * 100), score_rows=4096)


def test_full_size_paper_native_point():
    _full_size_check(wl.paper_native(), n_rows=256)


def test_full_size_long_horizon():
    # 93 600-token cache pruned to 9360: a cluster of eight selects, heavy-tailed scores
    _full_size_check(wl.long_horizon(), n_rows=256, score_rows=8192)


def test_full_size_batch4_14b():
    # four ragged streams, 40 heads, D_M = 5120, hidden 512 (two accumulator chunks per tile)
    _full_size_check(wl.batch4_14b(), n_rows=256, score_rows=2048)
