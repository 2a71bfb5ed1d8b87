"""Builds libgdn.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and the extension module of its Python binding.

    python -m paper_2607_14568_b200.build [--force] [--verbose]

nvcc cross-compiles without a GPU.  The CUDA runtime is linked statically and the
driver API is reached through the runtime's entry-point lookup, so the shared
object loads on a machine without a driver (symbols can be inspected there).
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libgdn.so")
CALL = os.path.join(PKG, "_call.so")               # native side of the Python binding
CALL_SRC = os.path.join(CSRC, "py_call.cpp")

NVCC_FLAGS = [
    "-std=c++17", "-O3", "-lineinfo",
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-Xcompiler", "-fPIC", "-shared", "-cudart", "static",
    "-I", os.path.join(ROOT, "include"), "-I", CSRC,
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(CALL) or os.path.getmtime(CALL_SRC) > os.path.getmtime(CALL):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh")) \
        + glob.glob(os.path.join(ROOT, "include", "*.h")) + [os.path.abspath(__file__)]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    _build_library(verbose)
    _build_call(verbose)
    return LIB


def _run(cmd, verbose: bool, what: str) -> None:
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
    if res.returncode != 0:
        raise RuntimeError(f"{cmd[0]} failed building {what}")


def _build_call(verbose: bool) -> None:
    """The binding's extension module: C++ against torch's headers, linked to the libgdn.so next to it."""
    import torch
    t = os.path.dirname(torch.__file__)
    tmp = CALL + f".tmp{os.getpid()}"
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    _run(["g++", "-std=c++17", "-O2", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
          "-I", os.path.join(ROOT, "include"), "-I", sysconfig.get_paths()["include"], "-I", os.path.join(cuda, "include"),
          "-isystem", os.path.join(t, "include"), "-isystem", os.path.join(t, "include", "torch", "csrc", "api", "include"),
          CALL_SRC, "-o", tmp, "-L", PKG, "-l:libgdn.so", "-Wl,-rpath,$ORIGIN",
          "-L", os.path.join(t, "lib"), "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"], verbose, "_call.so")
    os.replace(tmp, CALL)


def _build_library(verbose: bool) -> None:
    nvcc = os.environ.get("NVCC", "nvcc")
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", tmp] + sources()
    _run(cmd, verbose, "libgdn.so")
    os.replace(tmp, LIB)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
