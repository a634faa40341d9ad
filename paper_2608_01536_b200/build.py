"""Builds the C-ABI CUDA library in-tree, csrc/celty_host.cpp, csrc/celty_upload.cpp and csrc/*.cu -> libcelty.so (sm_100a only), and the module
behind the Python binding, csrc/celty_torch.cpp -> _celty_torch.so."""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libcelty.so")
SOURCES = [os.path.join(CSRC, "celty_host.cpp"), os.path.join(CSRC, "celty_upload.cpp"), os.path.join(CSRC, "celty_kernels.cu")]
HEADERS = [os.path.join(CSRC, "celty_internal.h"), os.path.join(CSRC, "celty_upload.h"), os.path.join(CSRC, "celty_signal.h"), os.path.join(CSRC, "celty_fused.cuh"), os.path.join(CSRC, "celty_direct.cuh"), os.path.join(CSRC, "celty_column.cuh"),
           os.path.join(ROOT, "include", "celty.h")]


# the binding's per-call functions, a CPython module that takes torch tensors
BINDING = os.path.join(HERE, "_celty_torch.so")
BINDING_SOURCE = os.path.join(CSRC, "celty_torch.cpp")


def _older(target, sources) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(f) > t for f in sources)


def _binding_outdated() -> bool:
    """The module is tied to the torch it was built against, which it names (TORCH_VERSION): file times do not tell."""
    import torch
    if _older(BINDING, [BINDING_SOURCE, os.path.join(ROOT, "include", "celty.h")]):
        return True
    with open(BINDING, "rb") as f:
        return b"built with torch %s\0" % torch.__version__.encode() not in f.read()


def needs_build() -> bool:
    return _older(LIB, SOURCES + HEADERS) or _binding_outdated()


def _build_binding() -> None:
    import sysconfig

    import torch
    base = os.path.join(os.path.dirname(torch.__file__))
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cuda = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include")
    subprocess.check_call(
        ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", '-DTORCH_VERSION="%s"' % torch.__version__, "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch._C._GLIBCXX_USE_CXX11_ABI,
         "-I", os.path.join(ROOT, "include"), "-I", sysconfig.get_paths()["include"], "-I", cuda,
         "-isystem", os.path.join(base, "include"), "-isystem", os.path.join(base, "include", "torch", "csrc", "api", "include"),
         BINDING_SOURCE, "-o", BINDING, "-L", HERE, "-l:libcelty.so", "-L", os.path.join(base, "lib"),
         "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python", "-Wl,-rpath,$ORIGIN"])


def build(force: bool = False, verbose: bool = False) -> str:
    if not (force or needs_build()):
        return LIB
    if force or _older(LIB, SOURCES + HEADERS):
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        cmd = [nvcc, "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
               "-Xcompiler", "-fPIC", "-shared", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
               "-o", LIB] + SOURCES
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        subprocess.check_call(cmd)
    if force or _binding_outdated():
        _build_binding()
    return LIB


if __name__ == "__main__":
    build(force=True, verbose="-v" in sys.argv)
    print(LIB)
