"""Build the CUDA library in-tree with nvcc for sm_100a, and the calls' host path beside it."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_HERE)
CSRC = os.path.join(_HERE, "csrc")
LIB = os.path.join(_HERE, "libsuffixspec.so")
SOURCES = ["build.cu", "append.cu", "speculate.cu", "query.cu", "device_memory.cpp"]


def call_path() -> str:
    """The module _call.  It is built against private headers of torch, so its name says for which torch (and Python):
    behind an upgrade of either the one that is there is not taken for the one that is needed."""
    import torch
    return os.path.join(_HERE, f"_call.{sys.implementation.cache_tag}-torch-{torch.__version__}.so")


def _newest_source() -> float:
    paths = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(_ROOT, "include", "suffixspec.h")]
    return max(os.path.getmtime(p) for p in paths)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile SOURCES into libsuffixspec.so (cross-compiles without a GPU) and csrc/call.cpp into the
    module _call.  Returns the library's path."""
    newest = _newest_source()

    def fresh(path):
        return not force and os.path.exists(path) and os.path.getmtime(path) >= newest

    if not fresh(LIB):
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
               "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(_ROOT, "include"), "-I", CSRC,
               "-cudart", "shared", "-Xlinker", "-z", "-Xlinker", "nodelete", "-o", LIB]   # (a thread of device_memory.cpp outlives dlclose)
        if verbose:
            cmd += ["-Xptxas", "-v"]
        cmd += [os.path.join(CSRC, f) for f in SOURCES]
        subprocess.check_call(cmd)
    if not fresh(call_path()):
        build_call()
    return LIB


def build_call() -> str:
    """Compile csrc/call.cpp into the module _call (host code, no nvcc).  Returns its path."""
    import torch
    from torch.utils.cpp_extension import include_paths
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    includes = [os.path.join(_ROOT, "include"), sysconfig.get_paths()["include"], os.path.join(cuda, "include"),
                *include_paths()]
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
    for path in includes:
        cmd += ["-isystem", path]
    cmd += [os.path.join(CSRC, "call.cpp"), "-L", lib, "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda", "-o", call_path()]
    subprocess.check_call(cmd)
    return call_path()


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
