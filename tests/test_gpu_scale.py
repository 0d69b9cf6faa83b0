"""The branch-free NVFP4 group scale against the IEEE division and reciprocal it stands for: every mantissa of a
reciprocal, every mantissa over 64 divisors, and 2.7e8 scales with zero, subnormal, infinite and NaN maxima among them."""
import os
import subprocess

import pytest

from paper_2605_09503_b200 import build

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_scale_equals_the_ieee_operations(tmp_path):
    exe = str(tmp_path / "scale_ieee")
    flags = [f for f in build.NVCC_FLAGS if f not in ("-Xcompiler", "-fPIC", "-Wall")]
    subprocess.run(["nvcc", *flags, "-I", build.CSRC, os.path.join(HERE, "scale_ieee.cu"), "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout
    assert out.split() == ["0", "0", "0"], out
