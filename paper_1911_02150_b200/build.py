"""Build the CUDA library in-tree: ``python -m paper_1911_02150_b200.build``.

nvcc cross-compiles for sm_100a without a GPU present.  The output,
``paper_1911_02150_b200/libmqa_decode.so``, exports the C ABI declared in
``include/mqa_decode.h``; the CUDA runtime is linked statically, so the library has no
dependency on which libcudart the host process loaded.
"""
from __future__ import annotations

import glob
import os
import shutil
import subprocess
import sys

from .binding import checked_call_path

PKG = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libmqa_decode.so")
INCLUDE = os.path.join(os.path.dirname(PKG), "include")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-O3", "-std=c++17", "-lineinfo",
    "-Xcompiler", "-fPIC", "-shared",
    "-cudart", "static",
]


def _nvcc() -> str:
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found: the CUDA library cannot be built")
    return exe


def _build_checked_call() -> None:
    import sysconfig
    import torch
    root = os.path.dirname(torch.__file__)
    path = checked_call_path()
    tmp = path + f".tmp{os.getpid()}"
    subprocess.check_call(
        ["g++", "-O2", "-shared", "-fPIC", "-std=c++17", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
         "-isystem", os.path.join(root, "include"), "-isystem", os.path.join(root, "include", "torch", "csrc", "api", "include"),
         "-isystem", os.path.join(os.path.dirname(os.path.dirname(_nvcc())), "include"), "-I", sysconfig.get_paths()["include"],
         os.path.join(CSRC, "checked_call.cpp"), "-o", tmp, "-L", PKG, "-l:" + os.path.basename(LIB), "-Wl,-rpath,$ORIGIN",
         "-L", os.path.join(root, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"])
    os.replace(tmp, path)


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    checked = checked_call_path()
    if not os.path.exists(LIB) or not os.path.exists(checked):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(checked))
    deps = glob.glob(os.path.join(CSRC, "*")) + glob.glob(os.path.join(INCLUDE, "*.h")) + [__file__]
    return any(os.path.getmtime(d) > t for d in deps)


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compile every ``csrc/*.cu`` into one shared library for sm_100a, and the binding's native half; returns the library's path."""
    if not force and not _stale():
        return LIB
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [_nvcc()] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-I", INCLUDE, "-o", tmp] + sources()
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)
    _build_checked_call()
    return LIB


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose="-v" in sys.argv))
