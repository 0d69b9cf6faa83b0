"""The native module beside the library: it binds to this package's library whatever else the loader could find."""
import os
import subprocess
import sys

from paper_2605_09503_b200 import build

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
