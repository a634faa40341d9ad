"""Builds the C-ABI CUDA library in-tree: csrc/*.cpp, csrc/*.cu -> libcelty.so (sm_100a only)."""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libcelty.so")
SOURCES = [os.path.join(CSRC, "celty_host.cpp"), os.path.join(CSRC, "celty_kernels.cu")]
HEADERS = [os.path.join(CSRC, "celty_internal.h"), os.path.join(CSRC, "celty_fused.cuh"), os.path.join(CSRC, "celty_direct.cuh"), os.path.join(CSRC, "celty_column.cuh"),
           os.path.join(ROOT, "include", "celty.h")]


def needs_build() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    return any(os.path.getmtime(f) > t for f in SOURCES + HEADERS)


def build(force: bool = False, verbose: bool = False) -> str:
    if not (force or needs_build()):
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
           "-Xcompiler", "-fPIC", "-shared", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
           "-o", LIB] + SOURCES
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
    subprocess.check_call(cmd)
    return LIB


if __name__ == "__main__":
    build(force=True, verbose="-v" in sys.argv)
    print(LIB)
