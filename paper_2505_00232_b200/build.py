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


def installed_torch():
    """(folder, what a module built against it is built for) of the installed torch, which is not imported for that; None if there is none."""
    spec = importlib.util.find_spec("torch")
    if spec is None:
        return None
    folder = spec.submodule_search_locations[0]
    spec = importlib.util.spec_from_file_location("_torch_version", os.path.join(folder, "version.py"))
    version = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(version)
    return folder, f"torch {version.__version__} {version.git_version} cuda {version.cuda} python {sysconfig.get_config_var('SOABI')}"


def build_native(force: bool = False):
    """The extension module of the binding, against the installed torch (which has loaded these libraries when the module is imported).  It uses
    C++ interfaces of torch and Python that change with their versions, so it holds their names and is built again when they differ.
    Without torch there is nothing to build it against, and nothing that would load it: packing and the C library need neither."""
    torch = installed_torch()
    if torch is None:
        return None
    folder, built_for = torch
    if not (force or _stale(NATIVE, ["native.cpp", HEADER])):
        with open(NATIVE, "rb") as f:
            if built_for.encode() + b"\0" in f.read():
                return NATIVE
    abi = subprocess.check_output([sys.executable, "-c", "import torch; print(int(torch.compiled_with_cxx11_abi()))"], text=True).strip()
    include = [os.path.join(folder, "include"), os.path.join(folder, "include", "torch", "csrc", "api", "include"), os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include"), sysconfig.get_paths()["include"]]
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden", "-D_GLIBCXX_USE_CXX11_ABI=" + abi, f'-DQL_BUILT_FOR="{built_for}"',
                           *("-I" + i for i in include), os.path.join(CSRC, "native.cpp"),
                           "-L" + os.path.join(folder, "lib"), "-ltorch_python", "-ltorch_cuda", "-ltorch_cpu", "-lc10_cuda", "-lc10", "-o", NATIVE])
    return NATIVE


def build(force: bool = False, verbose: bool = False) -> str:
    build_library(force, verbose)
    build_native(force)
    return LIB


def build_library(force: bool = False, verbose: bool = False) -> str:
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
