"""Builds the CUDA library (libtk.so) in-tree for sm_100a with nvcc.

    python -m paper_2302_01425_b200.build [--force] [--verbose] [--bounds]

--bounds builds the second target, libtk_bounds.so: the same sources with -DTK_DEBUG_BOUNDS, in which
the kernels of the default path range-check every index they form (a violation sets TK_FLAG_BOUNDS in
the status word and skips the access).  It stands in for a memory checker where none can be run.
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys

_PKG = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_PKG)
CSRC = os.path.join(_PKG, "csrc")
LIB = os.path.join(_PKG, "libtk.so")
LIB_BOUNDS = os.path.join(_PKG, "libtk_bounds.so")
BIND = os.path.join(_PKG, "_tk_bind.so")
BIND_SRC = os.path.join(CSRC, "host", "tk_bind.cpp")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-shared", "--threads", "0",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale(lib: str = LIB) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(
        os.path.join(_ROOT, "include", "*.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def build_bind(force: bool = False) -> str:
    """The C++ half of the binding (argument marshalling), against torch's headers and libraries."""
    header = os.path.join(_ROOT, "include", "tk.h")
    if not force and os.path.exists(BIND) and all(os.path.getmtime(f) <= os.path.getmtime(BIND) for f in (BIND_SRC, header)):
        return BIND
    import sysconfig
    import torch
    from torch.utils import cpp_extension
    base = os.path.join(os.path.dirname(torch.__file__))
    cuda = cpp_extension.CUDA_HOME or "/usr/local/cuda"
    tmp = BIND + f".tmp{os.getpid()}"
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", "-w",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}"]
    for d in [os.path.join(base, "include"), os.path.join(base, "include", "torch", "csrc", "api", "include"),
              sysconfig.get_paths()["include"], os.path.join(cuda, "include"), os.path.join(_ROOT, "include")]:
        cmd += ["-I", d]
    cmd += ["-o", tmp, BIND_SRC, "-L", os.path.join(base, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    subprocess.run(cmd, check=True)
    os.replace(tmp, BIND)
    return BIND


def build(force: bool = False, verbose: bool = False, bounds: bool = False) -> str:
    if not bounds:
        build_bind(force)
    lib = LIB_BOUNDS if bounds else LIB
    if not force and not _stale(lib):
        return lib
    nvcc = os.environ.get("NVCC", "nvcc")
    tmp = lib + f".tmp{os.getpid()}"
    cmd = [nvcc] + NVCC_FLAGS
    if bounds:
        cmd += ["-DTK_DEBUG_BOUNDS"]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += ["-I", os.path.join(_ROOT, "include"), "-I", CSRC, "-o", tmp] + sources()
    subprocess.run(cmd, check=True)
    os.replace(tmp, lib)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv, bounds="--bounds" in sys.argv))
