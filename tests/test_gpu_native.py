"""The native marshalling of the Python calls: errors keep their types, and the batches outlive the call that reads them."""
import sys
import threading

import pytest
import torch

from paper_2605_09503_b200 import binding as B
from paper_2605_09503_b200 import pipeline

pytestmark = pytest.mark.gpu
DEV = "cuda"


def test_an_output_that_does_not_fit_raises_out_of_memory():
    """2^27 x 2^20 outputs (2^48 bytes) of stretched one-row operands: the allocation fails, nothing is launched."""
    X = torch.zeros(1, 64, dtype=torch.bfloat16, device=DEV).expand(1 << 27, 64)
    wq = torch.zeros(1, 32, dtype=torch.uint8, device=DEV).expand(1 << 20, 32)
    one, byte = torch.ones(1, device=DEV), torch.zeros(512, dtype=torch.uint8, device=DEV)
    with pytest.raises(torch.OutOfMemoryError):
        B.linear(X, one, byte, byte, wq, byte, one, None, B.workspace(B.OP_GEMM, 1, 64, 8))


def test_batches_are_held_while_the_call_runs():
    """The interpreter lock is released around the call: another thread may empty the list of batches meanwhile."""
    x, w = (torch.ones(64, 512, dtype=torch.bfloat16, device=DEV) for _ in range(2))
    batches, counts, done = [x], set(), threading.Event()

    def watch():
        while not done.is_set():
            counts.add(sys.getrefcount(x))

    watcher = threading.Thread(target=watch)
    watcher.start()
    for _ in range(400):
        pipeline.calibrate(batches, w)
    done.set()
    watcher.join()
    torch.cuda.synchronize()
    assert max(counts) > sys.getrefcount(x)      # seen from the other thread: one reference more than the list's and ours
