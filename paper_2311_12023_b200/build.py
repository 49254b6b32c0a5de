"""Builds ``liblqlora.so`` (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and ``_fast.so`` (the native part of the binding)
with g++ against the installed torch."""
from __future__ import annotations

import glob
import os
import subprocess
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "liblqlora.so")
FAST = os.path.join(HERE, "_fast.so")
FAST_SRC = os.path.join(CSRC, "fast_binding.cpp")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    # IEEE arithmetic in the codec: no flush-to-zero, exact division and square root, no fast-math
    "--ftz=false", "--prec-div=true", "--prec-sqrt=true",
    "-shared", "-Xcompiler", "-fPIC",
]


def _stale(target: str, srcs) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(s) > t for s in srcs)


def build_fast() -> str:
    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
    for inc in (os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"), sysconfig.get_paths()["include"],
                os.path.join(cuda, "include")):
        cmd += ["-isystem", inc]
    cmd += ["-o", FAST, FAST_SRC, "-L" + os.path.join(root, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch", "-ltorch_python"]
    subprocess.run(cmd, check=True)
    return FAST


def build(force: bool = False, verbose: bool = False) -> str:
    header = os.path.join(HERE, "..", "include", "lqlora.h")
    if force or _stale(LIB, [s for s in glob.glob(os.path.join(CSRC, "*")) if s != FAST_SRC] + [header]):
        nvcc = os.environ.get("NVCC", "nvcc")
        cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", LIB, os.path.join(CSRC, "lqlora.cu")]
        subprocess.run(cmd, check=True)
    if force or _stale(FAST, [FAST_SRC, header]):
        build_fast()
    return LIB


if __name__ == "__main__":
    import sys
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
