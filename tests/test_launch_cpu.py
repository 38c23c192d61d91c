"""How the backward's launches are set up, on the host: launch_host.cu is the launch code over a stand-in for the CUDA
runtime that counts launches, refuses some and checks shared-memory limits."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SCENARIOS = ["contexts_in_turn", "refused_sorts", "clusters_stand_by", "eight_blocks_a_table", "tiles_of_the_sum"]


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    out = str(tmp_path_factory.mktemp("launch") / "launch_host")
    # the device code is not run: it is left unoptimised and never assembled
    subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=compute_100a", "-Xcicc", "-O0", "-O1", "-std=c++17",
                           "-cudart", "none", "-cudadevrt", "none", "-I", os.path.join(HERE, "..", "include"), "-o", out,
                           os.path.join(HERE, "launch_host.cu"), os.path.join(HERE, "launch_host_runtime.cpp")])
    return out


@pytest.mark.parametrize("scenario", SCENARIOS)
def test_launches(program, scenario):
    r = subprocess.run([program, scenario], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
