"""The offline kernels where their tables, chunks and lists end: candidate errors against the original-order kernel
on gathered columns (every scale range, non-finite values), candidate orders with ties across sort chunks against
the oracle, and the whole pass in one call against the separate calls."""
import numpy as np
import pytest
import torch

from oracle import pq_oracle as O
from paper_2605_09503_b200 import binding as B
from paper_2605_09503_b200 import pipeline

pytestmark = pytest.mark.gpu
DEV = "cuda"


def tensor_with_edges(rows, K, seed):
    """Rows over the whole bf16 exponent range, zero rows, subnormal ones, and single infinities and NaNs."""
    g = torch.Generator().manual_seed(seed)
    x = torch.randn(rows, K, generator=g) * torch.exp(3.0 * torch.randn(K, generator=g))
    kind = torch.arange(rows) % 9
    x[kind == 1] *= 1e30
    x[kind == 2] *= 1e-36          # absmax / Q and its reciprocal leave the normal range
    x[kind == 3] *= 1e-39
    x[kind == 4] = 0.0
    x[kind == 5, : K // 2] = 0.0
    x = x.to(torch.bfloat16)
    x[kind == 6, 3] = float("inf")
    x[kind == 7, 5] = float("nan")
    x[kind == 8] = -x[kind == 8].abs()
    return x.to(DEV)


def errors(x, fmt, ts, perms):
    K = x.shape[1]
    P = 1 if perms is None else perms.shape[0]
    err = torch.zeros(P, K // (16 if fmt[0] == B.KIND_NVFP4 else fmt[2]), dtype=torch.float64, device=DEV)
    B.pq_group_error(x, fmt, ts, perms, err, B.workspace(B.OP_GROUP_ERROR, x.shape[0], K, 0, P))
    return err.cpu().numpy()


@pytest.mark.parametrize("fmt,ts", [((B.KIND_NVFP4, 4, 16), t) for t in (0.01, 3e-38, 1e30, 0.0, float("inf"))]
                         + [((B.KIND_INT, b, g), 1.0) for b, g in ((2, 16), (3, 32), (4, 64), (4, 128), (8, 256))])
@pytest.mark.parametrize("rows,K,P", [(1, 512, 1), (150, 768, 3), (37, 3072, 8), (20, 16384, 2)])
def test_candidate_errors_match_the_original_order_on_gathered_columns(rows, K, P, fmt, ts):
    x = tensor_with_edges(rows, K, rows + K)
    tsd = torch.tensor([ts], device=DEV)
    perms = torch.stack([torch.randperm(K, generator=torch.Generator().manual_seed(p)) for p in range(P)]).to(DEV, torch.int32)
    got = errors(x, fmt, tsd, perms)
    for p in range(P):
        assert np.array_equal(got[p], errors(x[:, perms[p].long()].contiguous(), fmt, tsd, None)[0], equal_nan=True)


@pytest.mark.parametrize("fmt", [(B.KIND_NVFP4, 4, 16), (B.KIND_INT, 3, 32), (B.KIND_INT, 4, 64), (B.KIND_INT, 8, 256)])
@pytest.mark.parametrize("rows,K,P", [(6501, 512, 8), (6550, 512, 8), (912, 3072, 8), (900, 3072, 7), (901, 6400, 8), (288, 16384, 8), (294, 16384, 8)])
def test_candidate_errors_around_the_number_of_pairs_where_kernels_change(rows, K, P, fmt):
    """Both kernels of the candidate orders (pairs of 16-row chunks and orders on either side of the line on 148 SMs) against
    the original-order kernel on gathered columns."""
    x, ts = tensor_with_edges(rows, K, rows + K), torch.tensor([0.01], device=DEV)
    perms = torch.stack([torch.randperm(K, generator=torch.Generator().manual_seed(p)) for p in range(P)]).to(DEV, torch.int32)
    got = errors(x, fmt, ts, perms)
    for p in range(P):
        assert np.array_equal(got[p], errors(x[:, perms[p].long()].contiguous(), fmt, ts, None)[0], equal_nan=True)


@pytest.mark.parametrize("K", [8, 1024, 1032, 3080, 8192, 8200, 16384])
def test_orders_with_ties_across_chunks(K):
    rng = np.random.default_rng(K)
    sa, sw = rng.choice([0.0, 1.0, 2.0, 1e-300, 7.5], K), rng.choice([0.0, 1.0, 3.0], K)
    J = 3
    perms = torch.empty(J + 1, K, dtype=torch.int32, device=DEV)
    B.pq_select_perm(torch.from_numpy(sa).to(DEV), 10, torch.from_numpy(sw).to(DEV), 7, J, perms,
                     B.workspace(B.OP_SELECT_PERM, 0, K, 0, J + 1))
    assert np.array_equal(perms.cpu().numpy(), O.select_perm(sa, 10, sw, 7, J))


def separate_calls(batches, W, fmt, J, tau):
    (N, K), g = W.shape, 16 if fmt[0] == B.KIND_NVFP4 else fmt[2]
    zero = lambda *s, dtype=torch.float64: torch.zeros(s, dtype=dtype, device=DEV)
    sa, sw, aa, aw = zero(K), zero(K), zero(K, dtype=torch.float32), zero(K, dtype=torch.float32)
    for x, s, a in [(x, sa, aa) for x in batches] + [(W, sw, aw)]:
        B.pq_calib_stats(x, s, a, B.workspace(B.OP_CALIB_STATS, x.shape[0], K))
    ts_x, ts_w = zero(1, dtype=torch.float32), zero(1, dtype=torch.float32)
    B.pq_tensor_scale(aa, ts_x)
    B.pq_tensor_scale(aw, ts_w)
    perms = zero(J + 1, K, dtype=torch.int32)
    B.pq_select_perm(sa, sum(x.shape[0] for x in batches), sw, N, J, perms, B.workspace(B.OP_SELECT_PERM, 0, K, 0, J + 1))
    ex, ew, lam, E, sel = zero(J + 2, K // g), zero(J + 2, K // g), zero(2), zero(J + 2), zero(2, dtype=torch.int32)
    for x, ts, e in [(x, ts_x, ex) for x in batches] + [(W, ts_w, ew)]:
        ws = B.workspace(B.OP_GROUP_ERROR, x.shape[0], K, 0, J + 1)
        B.pq_group_error(x, fmt, ts, None, e[0:1], ws)
        B.pq_group_error(x, fmt, ts, perms, e[1:], ws)
    B.pq_error_weights(sa, sw, lam)
    B.pq_accept(ex, ew, lam, tau, sel[0:1], sel[1:2], E)
    wq, sf = zero(N, K // 2, dtype=torch.uint8), zero(B.sf_bytes(N, K, B.PQ_SF_TCGEN05), dtype=torch.uint8)
    ts_q = zero(1, dtype=torch.float32)
    B.pq_quant_weight(W, perms, sel, wq, sf, B.PQ_SF_TCGEN05, ts_q, B.workspace(B.OP_QUANT_WEIGHT, N, K))
    return dict(sumsq_a=sa, sumsq_w=sw, amax_a=aa, ts_x=ts_x, ts_w=ts_q, perms=perms, err_x=ex, err_w=ew, lam=lam, E=E, select=sel,
                wq=wq, sfw=sf)


@pytest.mark.parametrize("rows,N,K,fmt,J", [
    ([1], 8, 64, (B.KIND_NVFP4, 4, 16), 1),
    ([300, 17, 128, 129, 1], 392, 512, (B.KIND_INT, 4, 32), 5),
    ([40] * 63, 130, 128, (B.KIND_INT, 3, 64), 2),      # the weight closes a full list
    ([40] * 64, 130, 128, (B.KIND_NVFP4, 4, 16), 2),    # ... and comes alone
    ([130, 7] * 50, 520, 192, (B.KIND_NVFP4, 4, 16), 7),
    ([260, 500], 1000, 8256, (B.KIND_INT, 4, 16), 5),
])
def test_one_call_equals_the_separate_calls(rows, N, K, fmt, J):
    g = torch.Generator().manual_seed(len(rows) + K)
    scale = torch.exp(1.5 * torch.randn(K, generator=g))
    wide = [(torch.randn(r, K + 8 * (i % 3), generator=g)).to(DEV) for i, r in enumerate(rows)]
    batches = [(x[:, :K] * scale.to(DEV)).to(torch.bfloat16) if i % 2 else (x * 2).to(torch.bfloat16)[:, :K] for i, x in enumerate(wide)]
    W = (0.02 * torch.randn(N, K, generator=g)).to(DEV, torch.bfloat16)
    c = pipeline.calibrate(batches, W, fmt=fmt, J=J, tau=0.01)
    want = separate_calls(batches, W, fmt, J, 0.01)
    assert c.rows_a == sum(rows)
    for name, t in want.items():
        assert torch.equal(getattr(c, name), t), name


@pytest.mark.parametrize("rows,N,K,fmt,J", [([2500], 264, 3072, (B.KIND_NVFP4, 4, 16), 5),         # all SMs but one gather
                                            ([700], 136, 16384, (B.KIND_INT, 4, 128), 7)])          # ... in subsets of the orders
def test_weights_beside_a_full_chip(rows, N, K, fmt, J):
    test_one_call_equals_the_separate_calls(rows, N, K, fmt, J)


@pytest.mark.parametrize("n", [40, 26])      # 1440 slabs in two rounds; 936 in one, and the weight in one of its own
def test_rounds_of_many_slabs_equal_the_separate_calls(n):
    """More partial sums than one round's 64 MiB hold (1213 slabs of these widths)."""
    g = torch.Generator(device=DEV).manual_seed(n)
    x = torch.randn(4608, 3072, generator=g, device=DEV).mul_(3).to(torch.bfloat16)
    W = torch.randn(36864, 3072, generator=g, device=DEV).to(torch.bfloat16)
    batches = [x] * n
    c = pipeline.calibrate(batches, W, J=7)
    for name, t in separate_calls(batches, W, pipeline.NVFP4, 7, 0.0).items():
        assert torch.equal(getattr(c, name), t), name
