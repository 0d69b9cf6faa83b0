"""The native marshalling of the Python calls: errors keep their types."""
import pytest
import torch

from paper_2605_09503_b200 import binding as B

pytestmark = pytest.mark.gpu
DEV = "cuda"


def test_an_output_that_does_not_fit_raises_out_of_memory():
    """2^27 x 2^20 outputs (2^48 bytes) of stretched one-row operands: the allocation fails, nothing is launched."""
    X = torch.zeros(1, 64, dtype=torch.bfloat16, device=DEV).expand(1 << 27, 64)
    wq = torch.zeros(1, 32, dtype=torch.uint8, device=DEV).expand(1 << 20, 32)
    one, byte = torch.ones(1, device=DEV), torch.zeros(512, dtype=torch.uint8, device=DEV)
    with pytest.raises(torch.OutOfMemoryError):
        B.linear(X, one, byte, byte, wq, byte, one, None, B.workspace(B.OP_GEMM, 1, 64, 8))
