"""Build libspecverify.so (nvcc for sm_100a) and the native host path of binding.py (g++) in-tree, no JIT cache."""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
SRC = [os.path.join(HERE, "csrc", "specverify.cu")]
DEPS = [os.path.join(HERE, "csrc", f) for f in ("common.cuh", "verify.cuh", "rowops.cuh", "cut.cuh", "stream.cuh", "walk.cuh", "nodes.cuh", "trunc.cuh", "analysis.cuh")]
LIB = os.path.join(HERE, "libspecverify.so")
HEADERS = [os.path.join(ROOT, "include", "specverify.h")]


CALLS_SRC = os.path.join(HERE, "csrc", "torch_calls.cpp")
CALLS = os.path.join(HERE, "_torch_calls.so")


def stale(out: str = LIB, sources=tuple(SRC + DEPS + HEADERS)) -> bool:
    if not os.path.exists(out):
        return True
    t = os.path.getmtime(out)
    return any(os.path.getmtime(f) > t for f in sources)


def build_calls(force: bool = False) -> str:
    """The CPython module that marshals torch tensors into the C ABI."""
    if not (force or stale(CALLS, [CALLS_SRC] + HEADERS)):
        return CALLS
    import sysconfig
    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
           sysconfig.get_paths()["include"], os.path.join(cuda, "include"), os.path.join(ROOT, "include")]
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           *[f"-I{d}" for d in inc], "-o", CALLS, CALLS_SRC, f"-L{os.path.join(root, 'lib')}",
           "-ltorch_python", "-ltorch_cuda", "-ltorch_cpu", "-lc10_cuda", "-lc10"]
    subprocess.check_call(cmd)
    return CALLS


def build(force: bool = False, verbose: bool = False) -> str:
    build_calls(force)
    if not (force or stale()):
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
           "-Xcompiler", "-fPIC", "-shared", "-I", os.path.join(ROOT, "include"),
           "-o", LIB] + SRC
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    subprocess.check_call(cmd)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
