"""abi_host.cpp calls the library over a stand-in for the CUDA runtime: pointers that a call's kernels cannot use are refused on
the host, before anything is launched, and all others are taken; pooled lookups have their blocks in the order that suits their
bags."""
import glob
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2410_20046_b200", "csrc")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    out = str(tmp_path_factory.mktemp("abi") / "abi_host")
    # the device code is not run: it is left unoptimised and never assembled
    subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=compute_100a", "-Xcicc", "-O0", "-O1", "-std=c++17", "-t", "8",
                           "-cudart", "none", "-cudadevrt", "none", "-I", os.path.join(HERE, "..", "include"), "-o", out,
                           *sorted(glob.glob(os.path.join(CSRC, "*.cu"))),
                           *[os.path.join(HERE, f) for f in ("abi_host.cpp", "abi_host_runtime.cpp", "launch_host_runtime.cpp")]])
    return out


@pytest.mark.parametrize("scenario", ["sum", "forward", "rows", "empty", "order"])
def test_calls(program, scenario):
    r = subprocess.run([program, scenario], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
