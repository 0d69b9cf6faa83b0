"""The native module beside the library: it binds to this package's library whatever else the loader could find, and only
a module built against the running torch and Python is loaded."""
import os
import subprocess
import sys

import pytest
import torch

from paper_2605_09503_b200 import binding, build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_another_library_of_the_same_file_name_is_not_taken(tmp_path):
    """libpq.so is also the name of PostgreSQL's client library: a stand-in for it on the library path changes nothing."""
    build.build()
    source = tmp_path / "other.c"
    source.write_text("int PQlibVersion(void) { return 1; }\n")
    subprocess.run(["gcc", "-shared", "-fPIC", str(source), "-o", str(tmp_path / "libpq.so")], check=True)
    env = dict(os.environ, LD_LIBRARY_PATH=os.pathsep.join([str(tmp_path)] + os.environ.get("LD_LIBRARY_PATH", "").split(os.pathsep)))
    code = "from paper_2605_09503_b200 import binding as B; B.native().linear; B.native().calibrate"
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=env, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr


def test_a_module_built_against_another_torch_is_not_loaded(monkeypatch):
    """It reads tensors through that version's headers: after an upgrade the old binary must not be found."""
    build.build()
    monkeypatch.setattr(torch, "__version__", "0.0.0")
    monkeypatch.setattr(binding, "_native_module", None)
    with pytest.raises(ImportError, match="build"):
        binding.native()
