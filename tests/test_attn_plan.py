"""The attention kernels' schedule, checked on the host: the arithmetic that the launcher and the kernels share
(csrc/attn_plan.cuh) is compiled with a host compiler and run for many problems."""
import ctypes
import os
import random
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
FEW_PIECES = 8                      # the longest list that the merge of few pieces takes
PLAIN, SPLIT, OPENING = 0, 1, 2


@pytest.fixture(scope="module")
def planner(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("plan") / "plan.so")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-o", so, os.path.join(HERE, "attn_plan_host.cpp"),
                    "-I", os.path.join(cuda, "include"), "-I", os.path.join(ROOT, "include"),
                    "-L", os.path.join(cuda, "lib64"), "-lcudart_static", "-ldl", "-lrt", "-lpthread"], check=True)
    f = ctypes.CDLL(so).attn_plan
    f.restype = ctypes.c_int64
    out = np.zeros(1 << 20, dtype=np.int64)

    def plan(B, Lq, heads, has_chunk=True, max_ctas=148):        # 148: as on a B200, whatever device is here
        cu = [np.concatenate([[0], np.cumsum(x)]).astype(np.int64) for x in (B, Lq)]
        ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)
        n = f(len(B), ptr(cu[0]), ptr(cu[1]), heads, int(has_chunk), max_ctas, ptr(out), ctypes.c_int64(out.size))
        assert n > 0
        w = out[:n].tolist()
        head = dict(zip(("grid", "whole", "waves", "mode", "n_items", "longest"), w[:6]))
        runs = np.array(w[7:7 + 9 * w[6]], dtype=np.int64).reshape(-1, 9)
        at, merged = 7 + 9 * w[6] + 1, []
        for _ in range(head["n_items"]):
            k = w[at + 3]
            merged.append((w[at], w[at + 1], w[at + 2], w[at + 4:at + 4 + k]))
            at += 4 + k
        assert at == n
        return head, runs, merged
    return plan


def check(planner, B, Lq, heads, has_chunk=True, max_ctas=148):
    h, runs, merged = planner(B, Lq, heads, has_chunk, max_ctas)
    cu = np.concatenate([[0], np.cumsum(Lq)])
    assert 1 <= h["grid"] <= max_ctas
    tiles, slots = {}, {}
    per_cta = np.zeros(h["grid"], dtype=np.int64)
    pieces = {}
    for c, s, n, q0, sl, t0, t1, nt, piece in runs.tolist():
        assert 0 <= t0 < t1 <= nt and nt == -(-B[s] // 64) + (-(-Lq[s] // 64) if has_chunk else 0)
        assert sl == (2 if Lq[s] - q0 > 128 else 1)
        assert piece == (-1 if (t0, t1) == (0, nt) else 0 if t0 > 0 else 1)
        tiles.setdefault((s, n, q0), []).append((t0, t1, c))
        per_cta[c] += (t1 - t0) * (8 if sl == 2 else 7)
        if piece >= 0:
            assert (c, piece) not in pieces                      # a CTA has one slot for either kind of partial
            pieces[(c, piece)] = 1
    # every item's tiles are covered once, in order
    want = {(s, n, q0) for s in range(len(B)) for n in range(heads) for q0 in range(0, Lq[s], 256)}
    assert set(tiles) == want
    split = {}
    for (s, n, q0), rs in tiles.items():
        rs = sorted(rs)
        nt = -(-B[s] // 64) + (-(-Lq[s] // 64) if has_chunk else 0)
        assert rs[0][0] == 0 and rs[-1][1] == nt and all(a[1] == b[0] for a, b in zip(rs, rs[1:]))
        if len(rs) > 1:
            split[(int(cu[s]) + q0, n)] = (min(256, Lq[s] - q0), [c for _, _, c in rs])
    # the merge is told exactly the split items, their pieces in key order
    assert {(row, n): (rows, ctas) for row, rows, n, ctas in merged} == split and len(merged) == len(split)
    assert h["longest"] == max([len(c) for _, c in split.values()], default=0)
    if not h["whole"]:                                           # no CTA exceeds its even share by more than a tile
        assert per_cta.max() <= per_cta.sum() // h["grid"] + 1 + 8
    return h


def test_every_tile_is_covered_once(planner):
    rng = random.Random(7)
    lg = lambda lo, hi: int(round(lo * (hi / lo) ** rng.random()))
    for i in range(400):
        n = rng.choice([1, 1, 2, 3, 4])
        Lq = [lg(1, 3000) if rng.random() < 0.95 else 0 for _ in range(n)]
        if not any(Lq):
            continue
        has_chunk = rng.random() < 0.7
        B = [lg(1, 20000) if rng.random() < 0.9 or not has_chunk else 0 for _ in range(n)]
        check(planner, B, Lq, rng.choice([1, 2, 3, 5, 12, 24, 40]), has_chunk, rng.choice([148, 148, 31]))


@pytest.mark.parametrize("heads,Lq,nB,want", [
    # the sizes of test_attention_work_split: whole or split, pieces of the longest item (0: nothing merged)
    (1, 1, 1, dict(whole=1, longest=0, mode=SPLIT)), (2, 64, 128, dict(whole=1, longest=0, mode=SPLIT)),
    (3, 129, 500, dict(whole=0, longest=11, mode=SPLIT)),
    (1, 130, 2561, dict(whole=0, longest=44)), (1, 300, 2559, dict(whole=0, longest=45)),
    (2, 257, 1285, dict(whole=0, longest=26)),
    (3, 2000, 576, dict(whole=0, longest=7, mode=OPENING)),
    (40, 1100, 100, dict(whole=0, waves=1, longest=4, mode=PLAIN)),
    (6, 1900, 700, dict(whole=0, longest=4, mode=PLAIN)), (30, 515, 900, dict(whole=0, longest=3, mode=PLAIN)),
    # and of the peaked inputs: runs of two to three and of about ten tiles
    (2, 600, 3017, dict(whole=0, mode=SPLIT)), (2, 770, 12013, dict(whole=0, mode=PLAIN)),
    # whole items beside the line, and at the end of the carried rounding
    (140, 256, 448, dict(whole=1, longest=0, mode=OPENING)), (148, 256, 64 * 60, dict(whole=1, mode=OPENING)),
    (148, 256, 64 * 61, dict(whole=1, mode=PLAIN)), (148, 256, 1, dict(whole=1, mode=OPENING)), (90, 256, 448, dict(whole=0)),
])
def test_rules_of_the_split(planner, heads, Lq, nB, want):
    h = check(planner, [nB], [Lq], heads)
    assert {k: h[k] for k in want} == want
