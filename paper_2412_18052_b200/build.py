"""Builds the CUDA library in-tree with nvcc for sm_100a, and the CPython extension over it with the host
compiler (works without a GPU)."""
from __future__ import annotations

import os
import subprocess
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libgaf.so")
NATIVE = os.path.join(HERE, "_gaf_native.so")
NATIVE_SOURCE = os.path.join(CSRC, "gaf_native.cpp")
SOURCES = [os.path.join(CSRC, "gaf_api.cu"), os.path.join(CSRC, "gaf_static.cu")]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-shared", "-Xcompiler", "-fPIC", "-cudart", "shared"]


def _newest_source_mtime() -> float:
    newest = 0.0
    for root in (CSRC, os.path.join(os.path.dirname(HERE), "include")):
        for name in os.listdir(root):
            newest = max(newest, os.path.getmtime(os.path.join(root, name)))
    return newest


def _up_to_date(target: str) -> bool:
    return os.path.exists(target) and os.path.getmtime(target) >= _newest_source_mtime()


def _native_command(out: str) -> list:
    import torch
    from torch.utils.cpp_extension import include_paths, library_paths
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I" + sysconfig.get_paths()["include"], "-I" + os.path.join(cuda, "include")]
    cmd += ["-isystem" + p for p in include_paths()]
    cmd += ["-o", out, NATIVE_SOURCE, "-L" + HERE, "-l:libgaf.so", "-Wl,-rpath,$ORIGIN"]
    cmd += ["-L" + p for p in library_paths()] + ["-ltorch_python", "-ltorch_cpu", "-ltorch", "-lc10_cuda", "-lc10"]
    return cmd


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile ``libgaf.so`` and ``_gaf_native.so`` next to this file if they are missing or out of date."""
    if force or not _up_to_date(LIB):
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        tmp = LIB + f".{os.getpid()}.tmp"
        cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", tmp] + SOURCES
        subprocess.check_call(cmd)
        os.replace(tmp, LIB)
    if force or not _up_to_date(NATIVE):
        tmp = NATIVE + f".{os.getpid()}.tmp"
        subprocess.check_call(_native_command(tmp))
        os.replace(tmp, NATIVE)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
