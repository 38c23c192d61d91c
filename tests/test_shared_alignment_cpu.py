"""Dynamic shared memory begins behind a kernel's static shared memory, wherever that ends, at the alignment that its
declaration asks for: the kernels lay wider words over it than it is declared with, up to 16 bytes, and every declaration
has to say so."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2410_20046_b200", "csrc")
FILES = sorted(glob.glob(os.path.join(CSRC, "*.cu*")))


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_dynamic_shared_memory_is_declared_aligned(path):
    with open(path) as f:
        declared = [line.strip() for line in f if re.match(r"\s*extern __shared__", line)]
    assert [d for d in declared if "__align__(16)" not in d] == []
