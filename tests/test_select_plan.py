"""How selections and the row copies of small steps are handed to CTAs, checked on the host: csrc/select_plan.cuh is compiled with a
host compiler and run for many problems."""
import ctypes
import os
import random
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
SMS = 148                           # as on a B200, whatever device is here
BATCH = 4                           # pieces of 16 bytes a thread copies at once


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("plan") / "select_plan.so")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-o", so, os.path.join(HERE, "select_plan_host.cpp"),
                    "-I", os.path.join(cuda, "include"), "-I", os.path.join(ROOT, "include"),
                    "-L", os.path.join(cuda, "lib64"), "-lcudart_static", "-ldl", "-lrt", "-lpthread"], check=True)
    return ctypes.CDLL(so)


def arr(v):
    return np.array(v, dtype=np.int64).ctypes.data_as(ctypes.c_void_p)


def plan_copy(lib, T, B, sink, recent, chunks):
    out = np.zeros(3 + len(T) + 1, dtype=np.int64)
    i64 = ctypes.c_int64
    lib.plan_copy(len(T), arr(T), arr(B), i64(sink), i64(recent), i64(chunks), SMS, out.ctypes.data_as(ctypes.c_void_p))
    return int(out[0]), int(out[1]), out[3:]


def check_shares(lib, T, B, sink, recent, chunks):
    """Every stream with rows has CTAs, the GPU holds all of them at once, and none has much more to copy than an even share."""
    small, threads, first = plan_copy(lib, T, B, sink, recent, chunks)
    if not small:
        return False
    units = np.minimum(T, B) * chunks
    ctas = np.diff(first)
    assert first[0] == 0 and np.all(ctas[units > 0] > 0) and first[-1] <= SMS
    assert np.all(ctas == ctas[0]) or np.all(ctas[units == 0] == 0)
    # shares grow by a 64th until all fit; they fit at the latest when the even share leaves one more CTA a stream
    even = max(threads * BATCH, units.sum() / (SMS - len(T)))
    assert max(u / c for u, c in zip(units, ctas) if c) <= even * 65 / 64 + 1
    return True


@pytest.mark.parametrize("T,B,sink,recent,chunks", [
    ([3000] + [100] * 31, [3000] + [50] * 31, 5, 5, 192),         # one stream kept whole beside 31 short ones
    ([20000] + [60] * 31, [20000] + [30] * 31, 5, 5, 32),
    ([4000, 100, 100, 0], [3700, 50, 0, 0], 3600, 5, 192),        # mostly sink; nothing kept of one, an empty one
    ([512], [128], 4, 64, 16), ([1], [1], 0, 0, 8), ([3000], [3000], 0, 0, 192),
])
def test_shares_of_small_steps_follow_the_rows(lib, T, B, sink, recent, chunks):
    assert check_shares(lib, T, B, sink, recent, chunks)


def test_shares_of_many_small_steps(lib):
    rng = random.Random(3)
    lg = lambda lo, hi: int(round(lo * (hi / lo) ** rng.random()))
    small = 0
    for _ in range(2000):
        n = rng.choice([1, 2, 3, 8, 31, 32])
        T = [lg(1, 60000) if rng.random() < 0.9 else 0 for _ in range(n)]
        B = [rng.choice([t, t // 2, t // 10, 7]) for t in T]
        small += check_shares(lib, T, B, rng.choice([0, 5, 30000]), rng.choice([0, 9, 3000]), rng.choice([8, 16, 24, 192, 640]))
    assert small > 300


@pytest.mark.parametrize("T,B,sink,chunks,small", [
    # rows in and out around 44 MiB of always-kept ones and 64 MiB of all; more than one CTA selects
    ([3754], [3754], 0, 192, True), ([3755], [3755], 0, 192, False), ([4580], [4180], 4180 - 430, 192, True), ([4580], [4180], 4180 - 420, 192, False),
    ([6300], [5400], 2400, 192, True), ([6400], [5500], 2500, 192, False), ([4097], [1000], 0, 192, False),
])
def test_limits_of_small_steps(lib, T, B, sink, chunks, small):
    assert plan_copy(lib, T, B, sink, 0, chunks)[0] == small


def plan_selection(lib, M, covered=False):
    out = np.zeros(3, dtype=np.int64)
    T, i64 = [m + 5 for m in M], ctypes.c_int64
    lib.plan_selection(len(M), arr(T), arr([m // 2 + 5 for m in M]), i64(2), i64(3), int(covered), out.ctypes.data_as(ctypes.c_void_p))
    return out.tolist()


@pytest.mark.parametrize("M,ctas", [
    ([4096], 1), ([4097], 2), ([8193], 4), ([16385], 8), ([360448], 8),
    ([21840] * 15, 8), ([21840] * 16, 4), ([21840] * 32, 4), ([500] * 31 + [20000], 4),       # one wave
    ([180224] * 32, 4), ([500] * 31 + [180225], 8),                                            # the most four CTAs hold
])
def test_selecting_clusters_fit_on_the_gpu_at_once(lib, M, ctas):
    nc, per_cta, stream = plan_selection(lib, M)
    assert nc == ctas and not stream and per_cta * nc >= max(M) and per_cta <= 45056
    assert nc * len(M) <= (120 if nc == 8 else 128) or max(M) > nc // 2 * 45056


@pytest.mark.parametrize("M,ctas", [(16, 1), (17160, 1), (24576, 1), (24577, 2), (49152, 2), (49153, 4), (98305, 8), (360448, 8)])
def test_covered_selections_leave_few_sms_out(lib, M, ctas):
    """Beside a rolling cache's append copies, which take longer."""
    assert plan_selection(lib, [M], covered=True)[0] == ctas
