"""Integer fake-quant with an order against the streaming kernel on gathered columns, bit for bit: every scale range,
non-finite values, signed zeros, remainders of four rows, index vectors of any alignment."""
import pytest
import torch

from paper_2605_09503_b200 import binding as B
from test_gpu_offline_edges import tensor_with_edges

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("bits,group", [(2, 16), (3, 32), (4, 64), (4, 128), (8, 256)])
@pytest.mark.parametrize("rows,K,shift", [(1, 256, 0), (30, 768, 1), (150, 3072, 0), (7, 16384, 3)])
def test_order_matches_gathered_columns(rows, K, shift, bits, group):
    x = tensor_with_edges(rows, K, K + bits)
    x[:, 0] = -0.0
    perm = torch.randperm(K, generator=torch.Generator().manual_seed(rows))
    held = torch.zeros(K + 4, dtype=torch.int32, device=DEV)
    held[shift:shift + K] = perm.to(DEV)
    out, want = torch.zeros(rows, K + 8, dtype=torch.bfloat16, device=DEV)[:, :K], torch.zeros(rows, K, dtype=torch.bfloat16, device=DEV)
    B.pq_fakequant_int(x, (B.KIND_INT, bits, group), held[shift:shift + K], out)
    B.pq_fakequant_int(x[:, perm.to(DEV)].contiguous(), (B.KIND_INT, bits, group), None, want)
    assert torch.equal(out.contiguous().view(torch.int16), want.view(torch.int16))
