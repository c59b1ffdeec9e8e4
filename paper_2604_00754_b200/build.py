"""Builds the CUDA library in-tree with nvcc for sm_100a (no JIT cache, no torch extension)."""
from __future__ import annotations

import glob
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libsa_b200.so")
NATIVE = os.path.join(HERE, "_native.so")          # Python entry of the per-layer calls
NATIVE_SRC = os.path.join(CSRC, "sa_native.cpp")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "--use_fast_math", "-Xcompiler", "-fPIC", "-shared",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _older(target: str, deps) -> bool:
    return not os.path.exists(target) or \
        any(os.path.getmtime(f) > os.path.getmtime(target) for f in deps)


def stale() -> bool:
    headers = glob.glob(os.path.join(ROOT, "include", "*.h"))
    return _older(LIB, sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + headers)


def native_stale() -> bool:
    return _older(NATIVE, [NATIVE_SRC] + glob.glob(os.path.join(ROOT, "include", "*.h")))


def build_library(force: bool = False, verbose: bool = False) -> str:
    if not force and not stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB + ".%d.tmp" % os.getpid()
    cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + \
        ["-I", os.path.join(ROOT, "include"), "-I", CSRC, "-o", tmp] + sources()
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)
    return LIB


def build_native(force: bool = False) -> str:
    """The C++ module over torch's headers; links the CUDA library, so build that first."""
    if not force and not native_stale():
        return NATIVE
    import sysconfig

    import torch
    from torch.utils.cpp_extension import include_paths
    lib_dir = os.path.join(os.path.dirname(torch.__file__), "lib")
    tmp = NATIVE + ".%d.tmp" % os.getpid()
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-w",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI),
           "-I", os.path.join(ROOT, "include"), "-I", sysconfig.get_paths()["include"]]
    for path in include_paths("cuda"):
        cmd += ["-isystem", path]
    cmd += [NATIVE_SRC, "-o", tmp, "-L", HERE, "-l:libsa_b200.so", "-L", lib_dir, "-ltorch_python",
            "-ltorch_cuda", "-ltorch_cpu", "-lc10_cuda", "-lc10",
            "-Wl,-rpath,$ORIGIN", "-Wl,-rpath," + lib_dir]
    subprocess.check_call(cmd)
    os.replace(tmp, NATIVE)
    return NATIVE


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose="-v" in sys.argv))
    print(build_native(force="--force" in sys.argv))
