"""Bad arguments of the offline pass and of the native calls end in the documented status or AssertionError, before
anything is launched or allocated for them."""
import ctypes as C

import pytest
import torch

from paper_2605_09503_b200 import binding as B
from paper_2605_09503_b200 import build, pipeline

NULL, SHAPE, ALIGN, FORMAT, WORKSPACE = 1, 2, 3, 4, 5
P = 0x1000                       # stands for a device address, never touched


def calibrate(rows=(128,), ld=None, N=64, K=128, ldw=None, fmt=(B.KIND_INT, 4, 32), J=5, layout=B.PQ_SF_TCGEN05, n=None, x=P, w=P, codes=P,
              sumsq=P, ws=P, ws_bytes=None):
    build.build()
    L, n = B.lib(), len(rows) if n is None else n
    r, f = (C.c_int64 * max(1, len(rows)))(*rows), B.pq_format(*fmt)
    X, lds = (C.c_void_p * max(1, len(rows)))(*[x] * len(rows)), (C.c_int64 * max(1, len(rows)))(*[ld or K] * len(rows))
    need = L.pq_calibrate_workspace_bytes(n, r, N, K, f, J)
    outputs = [sumsq] + [P] * 10 + [codes, P]
    return L.pq_calibrate(n, X, r, lds, w, N, K, ldw or K, f, J, 0.0, layout, *outputs, ws, need if ws_bytes is None else ws_bytes, None)


@pytest.mark.parametrize("bad,status", [
    (dict(rows=()), SHAPE), (dict(n=-1), SHAPE), (dict(J=0), SHAPE), (dict(J=8), SHAPE), (dict(J=10 ** 9), SHAPE),
    (dict(rows=(128, 0)), SHAPE), (dict(rows=(-5,)), SHAPE), (dict(ld=64), SHAPE), (dict(ldw=64), SHAPE), (dict(N=0), SHAPE),
    (dict(K=0), SHAPE), (dict(K=144), SHAPE), (dict(K=16448), SHAPE), (dict(K=96), SHAPE),     # K % group, width, K % 64
    (dict(fmt=(2, 4, 32)), FORMAT), (dict(fmt=(B.KIND_INT, 4, 48)), FORMAT), (dict(fmt=(B.KIND_INT, 9, 32)), FORMAT), (dict(layout=7), FORMAT),
    (dict(x=None), NULL), (dict(w=None), NULL), (dict(sumsq=None), NULL), (dict(codes=None), NULL),
    (dict(x=P + 8), ALIGN), (dict(w=P + 8), ALIGN), (dict(ld=132), ALIGN), (dict(ldw=132), ALIGN), (dict(codes=P + 8), ALIGN), (dict(ws=P + 16), ALIGN),
    (dict(ws=None), WORKSPACE), (dict(ws_bytes=256), WORKSPACE),
])
def test_status_of_the_c_call(bad, status):
    assert calibrate(**bad) == status


def test_workspace_size_of_bad_sizes_is_zero():
    build.build()
    rows = (C.c_int64 * 1)(128)
    size = lambda n=1, N=64, K=128, kind=B.KIND_INT, J=5: B.lib().pq_calibrate_workspace_bytes(n, rows, N, K, B.pq_format(kind, 4, 32), J)
    assert size() > 0
    assert [size(n=0), size(N=0), size(K=0), size(kind=2), size(J=0), size(J=8), size(J=10 ** 9)] == [0] * 7


@pytest.mark.parametrize("rows,N,K,group,J", [([4608] * 64, 9216, 12288, 16, 7), ([4608] * 64, 3072, 3072, 16, 5), ([18432] * 200, 12288, 3072, 64, 5),
                                              ([200000, 5], 64, 3072, 16, 5), ([5, 200000], 64, 16384, 256, 1)])
def test_workspace_does_not_grow_with_the_number_of_batches(rows, N, K, group, J):
    """64 MiB of partial sums are enough for any number of batches, or what the largest tensor takes alone."""
    build.build()
    L, fmt = B.lib(), B.pq_format(B.KIND_INT, 4, group)
    size = lambda r, n_rows: L.pq_calibrate_workspace_bytes(len(r), (C.c_int64 * len(r))(*r), n_rows, K, fmt, J)
    alone = max(size([max(rows)], 1), size([1], N))
    assert size(rows, N) <= max((64 << 20) + 4 * K + 256, alone)


gpu = pytest.mark.gpu


def bf16(*shape):
    return torch.ones(*shape, dtype=torch.bfloat16, device="cuda")


@gpu
@pytest.mark.parametrize("kwargs,status", [
    (dict(J=0), SHAPE), (dict(J=-1), SHAPE), (dict(J=8), SHAPE), (dict(J=10 ** 9), SHAPE), (dict(fmt=(B.KIND_INT, 4, 0)), FORMAT),
    (dict(fmt=(B.KIND_INT, 4, 256)), SHAPE), (dict(fmt=(3, 4, 16)), FORMAT), (dict(sf_layout=7), FORMAT),
])
def test_status_of_the_python_call(kwargs, status):
    with pytest.raises(B.PqError) as e:
        pipeline.calibrate([bf16(64, 128)], bf16(64, 128), **kwargs)
    assert e.value.code == status


@gpu
def test_batches_of_the_python_call():
    w = bf16(64, 128)
    with pytest.raises(B.PqError) as e:
        pipeline.calibrate([], w)
    assert e.value.code == SHAPE
    with pytest.raises(B.PqError) as e:
        pipeline.calibrate([bf16(64, 128), bf16(0, 128)], w)
    assert e.value.code == NULL          # a tensor without rows has no address
    for bad in (bf16(64, 64), bf16(64, 128).float(), bf16(2, 64, 128), bf16(128, 64).t(), bf16(64, 128).cpu(), None):
        with pytest.raises(AssertionError):
            pipeline.calibrate([bf16(64, 128), bad], w)
    for batches in ((bf16(64, 128),), (bf16(64, 128) for _ in range(2)), bf16(3, 64, 128)):      # any sequence of batches
        assert pipeline.calibrate(batches, w).rows_a % 64 == 0


@gpu
def test_missing_workspace_and_inputs_of_other_forms():
    M, N, K = 64, 64, 128
    x, y, one = bf16(M, K), bf16(M, N), torch.ones(1, device="cuda")
    xq, wq = (torch.zeros(64, K // 2, dtype=torch.uint8, device="cuda") for _ in range(2))
    sf = torch.zeros(B.sf_bytes(128, K, B.PQ_SF_TCGEN05), dtype=torch.uint8, device="cuda")
    for call in (lambda: B.pq_gemm_w4a4(xq, sf, one, wq, sf, one, y, None), lambda: B.linear(x, one, xq, sf, wq, sf, one, None, None)):
        with pytest.raises(B.PqError) as e:
            call()
        assert e.value.code == WORKSPACE
    ws = B.workspace(B.OP_GEMM, M, K, N)
    for bad in (bf16(1, M, K), x.float(), bf16(K, M).t(), x.cpu()):
        with pytest.raises(AssertionError):
            B.linear(bad, one, xq, sf, wq, sf, one, None, ws)
    for bad in (bf16(1, M, N), bf16(M, N + 8), y.float(), bf16(N, M).t()):
        with pytest.raises(AssertionError):
            B.linear(x, one, xq, sf, wq, sf, one, bad, ws)
        with pytest.raises(AssertionError):
            B.pq_gemm_w4a4(xq, sf, one, wq, sf, one, bad, ws)
