"""The two four-row norm kernels on the same rows (few rows: four per block; many: sixteen per block) give the same
bytes, with subnormal, infinite and NaN rows among them, and those of the oracle on finite ones; subnormal values count
in the statistics and in the output."""
import numpy as np
import pytest
import torch

from oracle import pq_oracle as O
from paper_2605_09503_b200 import binding as B
from paper_2605_09503_b200 import inputs
from test_gpu_offline_edges import tensor_with_edges

pytestmark = pytest.mark.gpu
DEV = "cuda"


def run(h, kind, a, b, eps, perm, ts):
    M, K = h.shape
    codes = torch.empty(M, K // 2, dtype=torch.uint8, device=DEV)
    sf = torch.empty(B.sf_bytes(M, K, B.PQ_SF_LINEAR), dtype=torch.uint8, device=DEV)
    y = torch.empty(M, K, dtype=torch.bfloat16, device=DEV)
    B.pq_norm_quant_nvfp4(h, kind, a, b, eps, perm, torch.tensor([ts], device=DEV), codes, sf, B.PQ_SF_LINEAR, y)
    return codes, sf.view(M, K // 16), y.view(torch.int16)


@pytest.mark.parametrize("kind", [B.NORM_RMS, B.NORM_ADALN])
@pytest.mark.parametrize("M,K", [(2352, 1088), (2353, 1088), (2368, 3072), (2400, 64), (2500, 3520), (2500, 3584)])
def test_many_rows_equal_few_rows(kind, M, K):
    g = torch.Generator().manual_seed(K)
    h = tensor_with_edges(M, K, M + kind)
    a, b = torch.randn(K, generator=g).to(DEV), torch.randn(K, generator=g).to(DEV)
    perm = torch.randperm(K, generator=g).to(DEV, torch.int32)
    many = run(h, kind, a, b, 1e-6, perm, 0.01)
    for r in (0, 3, 1041, M - 37):
        few = run(h[r:r + 37].contiguous(), kind, a, b, 1e-6, perm, 0.01)
        for x, y in zip(many, few):
            assert torch.equal(x[r:r + 37], y)


@pytest.mark.parametrize("kind", [B.NORM_RMS, B.NORM_ADALN])
@pytest.mark.parametrize("M,K,with_perm", [(2400, 1088, True), (41, 1088, True), (41, 2048, False), (3, 16400, True)])
def test_subnormal_inputs_match_the_oracle(kind, M, K, with_perm):
    g = torch.Generator().manual_seed(M)
    h = (torch.randn(M, K, generator=g) * 1e-39).to(torch.bfloat16)       # all of them subnormal
    a, b = torch.rand(K, generator=g), torch.zeros(K)
    perm = torch.randperm(K, generator=g).to(torch.int32) if with_perm else None
    ts = 1e-38
    codes, sf, y = run(h.to(DEV), kind, a.to(DEV), b.to(DEV), 1e-6, None if perm is None else perm.to(DEV), ts)
    c_o, s_o, y_o = O.norm_quant_nvfp4(inputs.bits(h), kind, a.numpy(), b.numpy(), 1e-6, ts, None if perm is None else perm.numpy())
    assert s_o.any() and np.array_equal(codes.cpu().numpy(), c_o) and np.array_equal(sf.cpu().numpy(), s_o)
    assert np.array_equal(y.cpu().numpy().view(np.uint16), y_o)
