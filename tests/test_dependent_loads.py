"""A kernel that waits for the grid in front of it is resident while that grid still writes.  It must not read through the
non-coherent path, which is defined only for memory that nobody writes while the kernel lives: no __ldg, no ld.global.nc, and
no const __restrict__ parameter, whose plain loads the compiler may turn into one."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_09503_b200", "csrc")
WAIT = re.compile(r"wait_for_prior_grid\(\)|griddepcontrol\.wait")


def kernels(text):
    """(name, signature, body) of every __global__ function with a body."""
    for m in re.finditer(r"__global__[^;{]*?(\w+)\s*\((?=[^;{]*\{)", re.sub(r"__(launch_bounds|maxnreg|cluster_dims)__\([^)]*\)", "", text)):
        rest = m.string[m.end():]
        at = rest.index("{")
        depth, end = 0, at
        for end in range(at, len(rest)):
            depth += {"{": 1, "}": -1}.get(rest[end], 0)
            if depth == 0:
                break
        yield m.group(1), rest[:at], rest[at:end]


def dependents():
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        found += [(name, sig, body) for name, sig, body in kernels(text) if WAIT.search(body)]
    return found


DEPENDENTS = dependents()


def test_the_dependent_kernels_are_found():
    assert {"fold_partials", "gemm_w4a4_kernel", "quant_nvfp4_kernel", "norm_quant_quad_kernel", "group_error_gather"} <= {k[0] for k in DEPENDENTS}


@pytest.mark.parametrize("name,signature,body", DEPENDENTS, ids=[k[0] for k in DEPENDENTS])
def test_reads_are_coherent(name, signature, body):
    assert "__ldg(" not in body
    assert not re.search(r"const [\w ]+\*\s*__restrict__", signature)


def test_no_helper_loads_around_the_caches_coherence():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        with open(path) as f:
            assert ".nc." not in re.sub(r"//[^\n]*", "", f.read()), path
