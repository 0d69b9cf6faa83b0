"""Entry points called from several host threads at once, each on a stream of its own: no call fails because another
thread's launch takes another amount of shared memory, and every call returns the bytes of the call alone."""
import threading
import time

import pytest
import torch

from paper_2605_09503_b200 import binding as B
from paper_2605_09503_b200 import pipeline

pytestmark = pytest.mark.gpu
DEV = "cuda"
INT4_G64 = (B.KIND_INT, 4, 64)


def matrix(rows, K, seed):
    g = torch.Generator().manual_seed(seed)
    return (torch.randn(rows, K, generator=g) * torch.exp(torch.randn(K, generator=g))).to(torch.bfloat16).to(DEV)


def order(K):
    return torch.randperm(K, generator=torch.Generator().manual_seed(K)).to(torch.int32).to(DEV)


# each maker returns a call without arguments that returns its output tensors
def calibrate(K, fmt):
    x, w = matrix(130, K, 1), matrix(40, K, 2)

    def call():
        c = pipeline.calibrate([x, x], w, fmt=fmt)
        return c.sumsq_a, c.perms, c.err_x, c.err_w, c.E, c.select, c.wq, c.sfw
    return call


def sort(K):
    sa, sw = matrix(1, K, 3)[0].double().square(), matrix(1, K, 4)[0].double().square()
    perms, ws = torch.empty(6, K, dtype=torch.int32, device=DEV), B.workspace(B.OP_SELECT_PERM, 0, K, 0, 6)

    def call():
        B.pq_select_perm(sa, 10, sw, 7, 5, perms, ws)
        return (perms,)
    return call


def statistics(rows):
    x, ws = matrix(rows, 64, 5), B.workspace(B.OP_CALIB_STATS, rows, 64)

    def call():
        s, a = torch.zeros(64, dtype=torch.float64, device=DEV), torch.zeros(64, dtype=torch.float32, device=DEV)
        B.pq_calib_stats(x, s, a, ws)
        return s, a
    return call


def fakequant(K):
    x, perm = matrix(9, K, 6), order(K)
    out = torch.empty_like(x)

    def call():
        B.pq_fakequant_int(x, INT4_G64, perm, out)
        return (out,)
    return call


def producer(K, rows, launch):
    x, ts = matrix(rows, K, 7), torch.full((1,), 0.01, device=DEV)
    codes = torch.zeros(rows, K // 2, dtype=torch.uint8, device=DEV)
    sf = torch.zeros(B.sf_bytes(rows, K, B.PQ_SF_TCGEN05), dtype=torch.uint8, device=DEV)
    perm, a = order(K), torch.ones(K, device=DEV)

    def call():
        launch(x, perm, a, ts, codes, sf)
        return codes, sf
    return call


def gather(K):
    return producer(K, 9, lambda x, perm, a, ts, codes, sf: B.pq_quant_act_nvfp4_perm(x, perm, ts, codes, sf, B.PQ_SF_TCGEN05))


def norm(K, rows):
    return producer(K, rows, lambda x, perm, a, ts, codes, sf: B.pq_norm_quant_nvfp4(x, B.NORM_RMS, a, None, 1e-6, perm, ts, codes,
                                                                                     sf, B.PQ_SF_TCGEN05))


def hadamard(K):
    return producer(K, 9, lambda x, perm, a, ts, codes, sf: B.pq_hadamard_quant_nvfp4(x, perm, ts, codes, sf, B.PQ_SF_TCGEN05))


def linear(M, K, N):
    x, w = matrix(M, K, 8), matrix(N, K, 9)
    wq, sfw = torch.empty(N, K // 2, dtype=torch.uint8, device=DEV), torch.empty(B.sf_bytes(N, K, B.PQ_SF_TCGEN05), dtype=torch.uint8, device=DEV)
    ts = torch.empty(1, device=DEV)
    B.pq_quant_weight(w, None, None, wq, sfw, B.PQ_SF_TCGEN05, ts, B.workspace(B.OP_QUANT_WEIGHT, N, K))
    layer = pipeline.QuantLinear(wq, sfw, ts, torch.full((1,), 0.01, device=DEV), M)
    return lambda: (layer(x),)


PAIRS = {
    "calibrate": lambda: (calibrate(3072, pipeline.NVFP4), calibrate(12288, pipeline.NVFP4)),
    "calibrate_int": lambda: (calibrate(1024, INT4_G64), calibrate(8192, INT4_G64)),
    "sort": lambda: (sort(3072), sort(12288)),
    "statistics": lambda: (statistics(40000), statistics(60000)),         # slab sums of 313 and 469 slabs
    "fakequant": lambda: (fakequant(6400), fakequant(16384)),
    "gather": lambda: (gather(6400), gather(16384)),
    "norm_quad": lambda: (norm(6400, 9), norm(16384, 9)),
    "norm_group": lambda: (norm(2048, 2400), norm(3072, 2400)),
    "norm_wide": lambda: (norm(20480, 9), norm(32768, 9)),
    "hadamard": lambda: (hadamard(8192), hadamard(16384)),
    "linear": lambda: (linear(200, 512, 520), linear(520, 1088, 9480)),   # narrow and wide tiles: maps found per thread
}


SECONDS = 1.5  # long enough for a limit set by one thread to fall between another one's setting and its launch


@pytest.mark.parametrize("pair", list(PAIRS))
def test_threads(pair):
    calls = PAIRS[pair]() + PAIRS[pair]()         # two threads of either size, each with buffers of its own
    want = [[t.clone() for t in call()] for call in calls]
    torch.cuda.synchronize()
    failures, start = [], threading.Barrier(len(calls))

    def loop(call, expected):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                start.wait()
                end = time.monotonic() + SECONDS
                while time.monotonic() < end:
                    for _ in range(50):
                        got = call()
                    stream.synchronize()
                    assert all(torch.equal(g, w) for g, w in zip(got, expected))
        except Exception as e:
            failures.append(repr(e))

    threads = [threading.Thread(target=loop, args=(c, w)) for c, w in zip(calls, want)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures
