"""Builds the CUDA library in-tree: ``python -m paper_2607_06202_b200.build``."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libubep.so")
SOURCES = ["ubep_kernels.cu", "ubep_few.cu", "ubep_host.cu", "ubep_static.cu", "ubep_mapper.cu", "ubep_sync.cu", "ubep_sharded.cu"]
DEPENDS = SOURCES + ["ubep_common.cuh", "ubep_cluster.cuh", "ubep_launch.cuh", "ubep_few.cuh", "ubep_layout.cuh", "ubep_quant.cuh", "ubep_kernels.h", "ubep_sync.h", "ubep_sharded.h", "../../include/ubep.h"]
NATIVE = os.path.join(HERE, "_native.so")             # CPython module of the calls a layer makes every step
NATIVE_DEPENDS = ["ubep_py.cpp", "../../include/ubep.h"]


def up_to_date(target: str = LIB, depends=DEPENDS) -> bool:
    if not os.path.exists(target):
        return False
    t = os.path.getmtime(target)
    return all(os.path.getmtime(os.path.join(CSRC, d)) <= t for d in depends)


def build_native(force: bool = False) -> str:
    """g++ against the headers of the running torch and python; the symbols come from the loaded torch."""
    if not force and up_to_date(NATIVE, NATIVE_DEPENDS):
        return NATIVE
    import torch
    from torch.utils import cpp_extension
    cmd = [os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-fPIC", "-shared", "-o", NATIVE,
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
    cmd += [f"-isystem{d}" for d in cpp_extension.include_paths() + [sysconfig.get_paths()["include"]]]
    cmd += [f"-isystem{os.path.join(os.environ.get('CUDA_HOME', '/usr/local/cuda'), 'include')}"]
    cmd += [os.path.join(CSRC, "ubep_py.cpp")]
    cmd += [f"-L{d}" for d in cpp_extension.library_paths()]
    cmd += ["-lc10", "-lc10_cuda", "-ltorch", "-ltorch_cpu", "-ltorch_cuda", "-ltorch_python"]
    subprocess.run(cmd, check=True)
    return NATIVE


def build(force: bool = False, verbose: bool = False) -> str:
    """nvcc for sm_100a only; the library is a plain shared object with a C ABI.  Beside it the CPython module
    of the binding."""
    build_native(force)
    if not force and up_to_date():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, "-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a",
           "-Xcompiler", "-fPIC", "-shared", "-cudart", "static", "-o", LIB]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += [os.path.join(CSRC, s) for s in SOURCES]
    subprocess.run(cmd, check=True)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
