"""The Hadamard kernels with a warp or a team of warps per row over more rows than the grid has warps, with a last, partly filled group of rows."""
import numpy as np
import pytest
import torch

from oracle import pq_oracle as O
from paper_2605_09503_b200 import binding as B
from paper_2605_09503_b200 import inputs
from test_gpu_gemm import to_tc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K", [(2400, 3072), (4737, 1536), (9475, 768), (1, 3072), (3, 768),
                                 (1187, 6144), (2, 6144), (597, 12288), (1, 12288),
                                 (4739, 1024), (1, 1024), (2371, 2048), (1779, 4096)])
def test_rows_kernel_bit_exact(M, K):
    g = torch.Generator().manual_seed(M)
    x = (torch.randn(M, K, generator=g) * torch.exp(torch.randn(K, generator=g))).to(torch.bfloat16)
    perm = torch.randperm(K, generator=g).to(torch.int32)
    codes = torch.empty(M, K // 2, dtype=torch.uint8, device="cuda")
    sf = torch.full((B.sf_bytes(M, K, B.PQ_SF_TCGEN05),), 0xEE, dtype=torch.uint8, device="cuda")
    B.pq_hadamard_quant_nvfp4(x.to("cuda"), perm.to("cuda"), torch.tensor([0.02], device="cuda"), codes, sf, B.PQ_SF_TCGEN05)
    c_o, s_o, _, _ = O.hadamard_quant_nvfp4(inputs.bits(x), 0.02, perm.numpy())
    assert np.array_equal(codes.cpu().numpy(), c_o) and np.array_equal(sf.cpu().numpy(), to_tc(s_o))
