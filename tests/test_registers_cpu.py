"""What the compiler says of kernels that live by their registers."""
import os
import re
import shutil
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2410_20046_b200", "csrc")


def spill_loads(source):
    """{mangled kernel: bytes of spill loads}"""
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    r = subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-Xptxas", "-v", "-I",
                        os.path.join(CSRC, "..", "..", "include"), "-c", "-o", os.devnull, os.path.join(CSRC, source)],
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr
    found = re.findall(r"entry function '(\w+)'.*?(\d+) bytes spill loads", r.stdout + r.stderr, re.S)
    return {name: int(loads) for name, loads in found}


def test_one_index_forward_of_whole_warps():
    """Batches whose warps take 32 bags run in instances that do not pay for those of fewer bags: their widest spill, that of rows of 16
    features, is 116 bytes; with the number of bags as a value at run time rows of 20 to 48 features had 136."""
    # <lanes per row, pieces of a lane, exact, few bags a warp>
    whole = {k: v for k, v in spill_loads("fwd.cu").items() if re.search(r"fwd_onehot_kernelILi\d+ELi\d+ELb[01]E(Lb0E)?E", k)}
    assert len(whole) == 18
    assert max(whole.values()) <= 116, whole
