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


@pytest.mark.parametrize("rows,K", [(30, 768), (592, 512), (593, 512), (2501, 3072)])      # 148 and 149 blocks with an order
def test_chain_of_calls(rows, K):
    """Blocks start before the call in front has finished: a chain, in place in parts, gives what it gives call by call."""
    perm = torch.randperm(K, generator=torch.Generator().manual_seed(5)).to(DEV).to(torch.int32)
    fmt = (B.KIND_INT, 4, 64)

    def chain(wait):
        x, y = tensor_with_edges(rows, K, 5), torch.empty(rows, K, dtype=torch.bfloat16, device=DEV)
        for i in range(12):
            B.pq_fakequant_int(x, fmt, perm if i % 3 else None, y)
            if wait:
                torch.cuda.synchronize()
            B.pq_fakequant_int(y, fmt, perm if i % 2 else None, y)
            if wait:
                torch.cuda.synchronize()
            x, y = y, x
        return x

    assert torch.equal(chain(False).view(torch.int16), chain(True).view(torch.int16))
