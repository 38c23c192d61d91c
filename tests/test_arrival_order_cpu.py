"""The sums' last arriving warp adds what other warps have stored.  One lane counts the arrival and acquires; that the other
lanes' loads come behind it is the doing of a warp barrier (a shuffle orders no memory), which has to stand in between."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2410_20046_b200", "csrc")


@pytest.mark.parametrize("name", ["seg_groups.cuh", "seg_reduce.cuh"])
def test_warp_barrier_behind_every_arrival(name):
    with open(os.path.join(CSRC, name)) as f:
        code = re.sub(r"//.*", "", f.read())
    behind = [re.search(r"__syncwarp\(\)|\bfold\((?!\s*int )", code[m.end():]) for m in re.finditer(r"= arrive\(", code)]
    behind += [re.search(r"__syncwarp\(\)|\bfold\((?!\s*int )", code[m.end():]) for m in re.finditer(r"arrive\(arrived\)", code)]
    assert len(behind) >= 2 and all(b and b.group().startswith("__syncwarp") for b in behind)
