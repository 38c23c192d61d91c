"""Builds the CUDA library in-tree with nvcc for sm_100a, and the native half of the Python binding with g++.

    python -m paper_2410_20046_b200.build [--force] [--verbose]
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libdqrm_b200.so")
NATIVE_SRC = os.path.join(CSRC, "binding.cpp")
NATIVE = os.path.join(HERE, "_dqrm_native.so")
NATIVE_FOR = NATIVE + ".for"          # what the module was built for

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-O3", "-lineinfo", "-std=c++17",
    "-Xcompiler", "-fPIC", "-shared",
    "-I", os.path.join(ROOT, "include"),
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + [os.path.join(ROOT, "include", "dqrm.h")]
    return any(os.path.getmtime(d) > os.path.getmtime(LIB) for d in deps)


def _native_for() -> str:
    """The Python and the torch that a module built now could be loaded by."""
    from importlib import metadata

    return f"python {sys.implementation.cache_tag} torch {metadata.version('torch')}\n"


def _native_stale() -> bool:
    deps = [NATIVE_SRC, os.path.join(ROOT, "include", "dqrm.h")]
    if not os.path.exists(NATIVE) or any(os.path.getmtime(d) > os.path.getmtime(NATIVE) for d in deps):
        return True
    try:
        with open(NATIVE_FOR) as f:
            return f.read() != _native_for()
    except OSError:
        return True


def build_native() -> None:
    import sysconfig

    import torch
    from torch.utils import cpp_extension

    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    includes = [os.path.join(ROOT, "include"), sysconfig.get_paths()["include"], os.path.join(cuda, "include"),
                *cpp_extension.include_paths()]
    tmp = NATIVE + f".tmp{os.getpid()}"
    # torch's libraries are loaded by `import torch`, which comes before the module's import
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}", *[f"-I{i}" for i in includes],
           "-o", tmp, NATIVE_SRC, f"-L{os.path.join(os.path.dirname(torch.__file__), 'lib')}",
           "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    subprocess.check_call(cmd)
    os.replace(tmp, NATIVE)
    with open(NATIVE_FOR, "w") as f:
        f.write(_native_for())


def build(force: bool = False, verbose: bool = False) -> str:
    if force or _native_stale():
        build_native()
    if not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "nvcc")
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [nvcc, *NVCC_FLAGS, *(["-Xptxas", "-v"] if verbose else []), "-o", tmp, *sources()]
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
