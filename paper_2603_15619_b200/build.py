"""Builds the CUDA library (libmoda_b200.so, nvcc for sm_100a) and the host path of its hot calls (_host.<abi>.so, g++) in-tree."""
from __future__ import annotations

import os
import subprocess
import sys

from . import binding
from .binding import HOST_PATH as HOST

PKG = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libmoda_b200.so")
SOURCES = [os.path.join(CSRC, "moda_api.cu")]
HOST_SOURCE = os.path.join(CSRC, "moda_host.cpp")
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-O3", "-std=c++17", "-lineinfo",
    "-Xcompiler", "-fPIC", "-shared",
    "-Xptxas", "-v",
    "--expt-relaxed-constexpr",
]


def _deps():
    out = [os.path.join(PKG, "..", "include", "moda.h")]
    for f in os.listdir(CSRC):
        if f.endswith((".cu", ".cuh", ".h")):
            out.append(os.path.join(CSRC, f))
    return out


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile if the library is missing or older than any source. Returns the .so path."""
    stale = not os.path.exists(LIB) or any(os.path.getmtime(d) > os.path.getmtime(LIB) for d in _deps())
    if force or stale:
        nvcc = os.environ.get("NVCC", "nvcc")
        tmp = LIB + f".tmp{os.getpid()}"
        cmd = [nvcc] + NVCC_FLAGS + ["-o", tmp] + SOURCES + ["-lcudart"]
        res = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or res.returncode != 0:
            sys.stderr.write(res.stdout + res.stderr)
        if res.returncode != 0:
            raise RuntimeError("nvcc failed building libmoda_b200.so")
        with open(os.path.join(PKG, "build_ptxas.log"), "w") as f:
            f.write(res.stdout + res.stderr)
        os.replace(tmp, LIB)
    return LIB


def build_host(force: bool = False, verbose: bool = False) -> str:
    """The CPython extension that moves the hot calls' host work out of Python (csrc/moda_host.cpp). Returns the .so path,
    which another Python or torch does not look for."""
    deps = (HOST_SOURCE, os.path.join(PKG, "..", "include", "moda.h"))
    if force or not os.path.exists(HOST) or any(os.path.getmtime(d) > os.path.getmtime(HOST) for d in deps):
        import sysconfig

        import torch
        root = os.path.dirname(torch.__file__)
        cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
        include = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
                   os.path.join(cuda, "include"), sysconfig.get_paths()["include"]]
        tmp = HOST + f".tmp{os.getpid()}"
        cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
        cmd += [f"-I{d}" for d in include] + ["-o", tmp, HOST_SOURCE, "-L" + os.path.join(root, "lib")]
        cmd += ["-ltorch_python", "-ltorch", "-ltorch_cpu", "-ltorch_cuda", "-lc10", "-lc10_cuda"]
        res = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or res.returncode != 0:
            sys.stderr.write(res.stdout + res.stderr)
        if res.returncode != 0:
            raise RuntimeError(f"g++ failed building {HOST}")
        os.replace(tmp, HOST)
    if isinstance(binding._host, binding._NoHost):            # calls of this process that came before the build
        binding._host = None
    return HOST


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
    print(build_host(force="--force" in sys.argv, verbose=True))
