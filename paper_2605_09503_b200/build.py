"""Build the CUDA library in-tree: csrc/*.cu -> paper_2605_09503_b200/libpq.so (sm_100a only).

nvcc cross-compiles without a GPU.  The runtime is linked statically and the driver entry
points are resolved at run time, so the library loads on a machine without a driver too.
"""
import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libpq.so")
# What the native module asks the loader for.  libpq.so is also the name of PostgreSQL's client library; under a name of its
# own the library is found among the loaded ones (binding.lib() loads it by path first) and nothing is searched.
SONAME = "libpq_permuquant_b200.so"
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-Xcompiler", "-Wall", "--fmad=false", "-cudart", "static"]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _older(target, deps):
    return not os.path.exists(target) or any(os.path.getmtime(d) > os.path.getmtime(target) for d in deps)


def _stale():
    return _older(LIB, sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + [os.path.join(HERE, "..", "include", "pq.h"), __file__])


def native_path() -> str:
    """The marshalling of the runtime calls (torch headers, no device code).  It holds one torch version's and one Python's
    ABI, so both are part of its name: after an upgrade the old binary is not found, and build() makes the new one."""
    import torch

    return os.path.join(HERE, f"_pq_native-torch{torch.__version__}{sysconfig.get_config_var('EXT_SUFFIX')}")


def build_native(force: bool = False) -> str:
    src, target = os.path.join(CSRC, "pq_native.cpp"), native_path()
    if force or _older(target, [src, LIB, __file__]):
        import torch

        root = os.path.dirname(torch.__file__)
        subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-Wall", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
                        f"-I{root}/include", f"-I{root}/include/torch/csrc/api/include", f"-I{sysconfig.get_paths()['include']}",
                        "-I/usr/local/cuda/include", src, "-o", target, f"-L{HERE}", "-l:libpq.so", f"-L{root}/lib",
                        "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"], check=True)
    return target


def build(force: bool = False, verbose: bool = False) -> str:
    if force or _stale():
        objs = []
        for src in sources():
            obj = src[:-3] + ".o"
            cmd = ["nvcc", *NVCC_FLAGS, "-c", src, "-o", obj]
            if verbose:
                cmd.insert(1, "-Xptxas=-v")
            subprocess.run(cmd, check=True)
            objs.append(obj)
        subprocess.run(["nvcc", "-Wno-deprecated-gpu-targets", "-shared", "-cudart", "static", "-Xlinker", f"-soname={SONAME}", "-o", LIB, *objs, "-ldl",
                        "-lpthread", "-lrt"], check=True)
    build_native(force)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
