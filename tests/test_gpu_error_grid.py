"""The persistent error kernel is one block per SM and its work is cut into equal shares: a block more than there are SMs starts when
another has ended and ends last.  The launched grid is read from a captured graph."""
import pytest
import torch

from paper_2605_09503_b200 import binding as B
from paper_2605_09503_b200 import pipeline

pytestmark = pytest.mark.gpu
DEV = "cuda"


def launched_blocks(graph, name):
    """Blocks of every kernel node of a captured graph whose name holds `name`."""
    from cuda.bindings import driver

    def ok(result):
        assert result[0] == driver.CUresult.CUDA_SUCCESS, result[0]
        return result[1:]

    handle = driver.CUgraph(graph.raw_cuda_graph())
    nodes, _ = ok(driver.cuGraphGetNodes(handle, ok(driver.cuGraphGetNodes(handle, 0))[1]))
    found = []
    for node in nodes:
        if ok(driver.cuGraphNodeGetType(node))[0] != driver.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL:
            continue
        p = ok(driver.cuGraphKernelNodeGetParams(node))[0]
        label = ok(driver.cuFuncGetName(p.func))[0] if int(p.func) else ok(driver.cuKernelGetName(p.kern))[0]
        if name.encode() in label:
            found.append(p.gridDimX * p.gridDimY * p.gridDimZ)
    return found


@pytest.mark.parametrize("K", [3072, 6144, 8192, 12288, 16384])
@pytest.mark.parametrize("fmt", [pipeline.NVFP4, (B.KIND_INT, 4, 64)])
def test_a_block_per_sm_at_most(K, fmt):
    g = torch.Generator(device=DEV)
    g.manual_seed(K)
    x, w = (torch.randn(n, K, device=DEV, generator=g).to(torch.bfloat16) for n in (900, 136))
    pipeline.calibrate([x], w, fmt=fmt)                       # attributes are set outside the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        pipeline.calibrate([x], w, fmt=fmt)
    blocks = launched_blocks(graph, "group_error_gather")
    assert len(blocks) == 1
    assert blocks[0] <= torch.cuda.get_device_properties(0).multi_processor_count
