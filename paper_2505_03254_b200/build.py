"""Builds the C-ABI CUDA library in-tree with nvcc for sm_100a, and the extension module beside it."""
from __future__ import annotations

import glob
import os
import subprocess
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(_HERE), "include")
LIB = os.path.join(_HERE, "libprom.so")
NATIVE = os.path.join(_HERE, "_native.so")
NATIVE_SOURCE = os.path.join(CSRC, "native.cpp")


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))
                  + glob.glob(os.path.join(INCLUDE, "*.h")))


def _native_sources():
    # the extension is compiled against the header's structures and signatures
    return [NATIVE_SOURCE] + sorted(glob.glob(os.path.join(INCLUDE, "*.h")))


def _older(target: str, sources) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(f) > os.path.getmtime(target) for f in sources)


def needs_build() -> bool:
    return _older(LIB, _sources()) or _older(NATIVE, _native_sources())


def _build_lib(verbose: bool) -> None:
    """nvcc -gencode arch=compute_100a,code=sm_100a ... -shared -> libprom.so"""
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-shared", "-Xcompiler", "-fPIC", "-Xlinker", "-soname=libprom.so", "-I", INCLUDE, "-I", CSRC,
           "-o", tmp, os.path.join(CSRC, "api.cu")]
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)


def _build_native() -> None:
    """g++ ... csrc/native.cpp -> _native.so, which finds libprom.so beside itself."""
    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    tmp = NATIVE + f".tmp{os.getpid()}"
    includes = [INCLUDE, os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
                sysconfig.get_paths()["include"], os.path.join(cuda, "include")]
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
    for d in includes:
        cmd += ["-I", d]
    cmd += [NATIVE_SOURCE, "-o", tmp, "-L", _HERE, "-l:libprom.so", "-Wl,-rpath,$ORIGIN", "-L", os.path.join(root, "lib"),
            "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    subprocess.check_call(cmd)
    os.replace(tmp, NATIVE)


def build(force: bool = False, verbose: bool = False) -> str:
    """Builds what is older than its sources; returns the path of the C-ABI library."""
    if force or _older(LIB, _sources()):
        _build_lib(verbose)
    if force or _older(NATIVE, _native_sources()):
        _build_native()
    return LIB


if __name__ == "__main__":
    import sys
    print(build(force=True, verbose="-v" in sys.argv))
