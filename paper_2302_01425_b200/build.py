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
import warnings

_PKG = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_PKG)
CSRC = os.path.join(_PKG, "csrc")
LIB = os.path.join(_PKG, "libtk.so")
LIB_BOUNDS = os.path.join(_PKG, "libtk_bounds.so")
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


def bind_path() -> str:
    """Where the C++ half of the binding lies.  It reads tensors by the layout of one torch and objects by that of one Python,
    and neither is stable: both versions are in its name, and another's is not picked up."""
    import torch
    return os.path.join(_PKG, f"_tk_bind.{sys.implementation.cache_tag}-torch{torch.__version__}.so")


def build_bind(force: bool = False) -> str:
    """The C++ half of the binding (argument marshalling), against torch's headers and libraries."""
    out = bind_path()
    header = os.path.join(_ROOT, "include", "tk.h")
    if not force and os.path.exists(out) and all(os.path.getmtime(f) <= os.path.getmtime(out) for f in (BIND_SRC, header)):
        return out
    import sysconfig
    import torch
    from torch.utils import cpp_extension
    base = os.path.join(os.path.dirname(torch.__file__))
    cuda = cpp_extension.CUDA_HOME or "/usr/local/cuda"
    tmp = out + f".tmp{os.getpid()}"
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", "-w",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}"]
    for d in [os.path.join(base, "include"), os.path.join(base, "include", "torch", "csrc", "api", "include"),
              sysconfig.get_paths()["include"], os.path.join(cuda, "include"), os.path.join(_ROOT, "include")]:
        cmd += ["-I", d]
    cmd += ["-o", tmp, BIND_SRC, "-L", os.path.join(base, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    subprocess.run(cmd, check=True)
    os.replace(tmp, out)
    return out


def build(force: bool = False, verbose: bool = False, bounds: bool = False) -> str:
    lib = LIB_BOUNDS if bounds else LIB
    if force or _stale(lib):
        _build_library(lib, verbose, bounds)
    if not bounds:
        try:
            build_bind(force)
        except (ImportError, OSError, subprocess.CalledProcessError) as e:      # the library serves without it
            warnings.warn(f"the C++ half of the binding could not be built ({e}): calls will go through ctypes, "
                          "8 us of host time each", RuntimeWarning, stacklevel=2)
    return lib


def _build_library(lib: str, verbose: bool, bounds: bool) -> None:
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


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv, bounds="--bounds" in sys.argv))
