"""Builds ``liblqlora.so`` (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and ``_fast`` (the native part of the binding, an
extension module of this Python) with g++ against the installed torch."""
from __future__ import annotations

import glob
import os
import subprocess
import sysconfig
import warnings

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "liblqlora.so")
FAST = os.path.join(HERE, "_fast" + sysconfig.get_config_var("EXT_SUFFIX"))
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


def built_for() -> str:
    """What the native part of the binding has to be compiled for: it reads torch's and Python's own structures."""
    import torch
    return f"torch {torch.__version__} python {sysconfig.get_config_var('SOABI')}"


def fast_stale() -> bool:
    if _stale(FAST, [FAST_SRC, os.path.join(HERE, "..", "include", "lqlora.h")]):
        return True
    with open(FAST, "rb") as f:
        return built_for().encode() not in f.read()


def build_fast() -> str:
    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", f'-DLQLORA_BUILT_FOR="{built_for()}"', f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
    for inc in (os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"), sysconfig.get_paths()["include"],
                os.path.join(cuda, "include")):
        cmd += ["-isystem", inc]
    cmd += ["-o", FAST, FAST_SRC, "-L" + os.path.join(root, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch", "-ltorch_python"]
    subprocess.run(cmd, check=True)
    return FAST


def build(force: bool = False, verbose: bool = False) -> str:
    if force or _stale(LIB, [s for s in glob.glob(os.path.join(CSRC, "*")) if s != FAST_SRC] + [os.path.join(HERE, "..", "include", "lqlora.h")]):
        nvcc = os.environ.get("NVCC", "nvcc")
        cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", LIB, os.path.join(CSRC, "lqlora.cu")]
        subprocess.run(cmd, check=True)
    if force or fast_stale():
        try:
            build_fast()
        except (OSError, subprocess.CalledProcessError) as e:      # no C++ compiler, no headers: the binding goes without it, and says so
            warnings.warn(f"the native part of the binding was not built: {e}", RuntimeWarning)
    return LIB


if __name__ == "__main__":
    import sys
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
