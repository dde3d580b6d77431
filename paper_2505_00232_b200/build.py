"""Builds libqlinear.so in-tree with nvcc for sm_100a (cross-compiles without a GPU), and the native half of the Python binding with g++."""
from __future__ import annotations

import importlib.util
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libqlinear.so")
NATIVE = os.path.join(HERE, "_native.so")
HEADER = os.path.join("..", "..", "include", "qlinear.h")
SOURCES = ["qlinear.cu", "pack.cpp"]
DEPS = SOURCES + ["layout.h", "dequant.cuh", "sm100_ptx.cuh", "embed.cuh", "gemv.cuh", "gemv_rows.cuh", "gemv_cols.cuh", "gemv_a8.cuh", "kv.cuh", "gemv_stream.cuh", "gemm.cuh", "gemm_mid.cuh", "gemm_rows.cuh", "gemm_pair.cuh", "gemm_pair_ta.cuh", "gemm_narrow.cuh", "norm.cuh", "rope.cuh", HEADER]


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(os.path.join(CSRC, d)) > t for d in deps)


def build_native(force: bool = False) -> str:
    """The extension module of the binding, against the installed torch (which has loaded these libraries when the module is imported)."""
    if not (force or _stale(NATIVE, ["native.cpp", HEADER])):
        return NATIVE
    torch = importlib.util.find_spec("torch").submodule_search_locations[0]
    include = [os.path.join(torch, "include"), os.path.join(torch, "include", "torch", "csrc", "api", "include"), os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include"), sysconfig.get_paths()["include"]]
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden", *("-I" + i for i in include), os.path.join(CSRC, "native.cpp"),
                           "-L" + os.path.join(torch, "lib"), "-ltorch_python", "-ltorch_cuda", "-ltorch_cpu", "-lc10_cuda", "-lc10", "-o", NATIVE])
    return NATIVE


def build(force: bool = False, verbose: bool = False) -> str:
    build_native(force)
    if not (force or _stale(LIB, DEPS)):
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
           "-Xcompiler", "-fPIC,-O3,-fopenmp,-falign-functions=64,-falign-loops=64", "-shared", "-cudart", "static",
           "-o", LIB] + [os.path.join(CSRC, s) for s in SOURCES] + ["-lgomp"]
    cmd[1:1] = os.environ.get("QL_EXTRA_NVCC_FLAGS", "").split()   # extra compiler flags, e.g. -DNAME for an experiment build
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    subprocess.check_call(cmd)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
