"""GPU parity of the pooled forward at its edges: bags around the batches of four and eight rows and the 32 indices that a
warp holds, batches on either side of the mean length at which a warp takes a bag, every row width class, with codes and
without.  FP64 sums in bag order have one value, so outputs are compared bit for bit."""
import numpy as np
import pytest

from dqrm_inputs import workloads as W
from gpu_util import Case, bit_equal

pytestmark = pytest.mark.gpu

LENGTHS = {
    "short": [0, 1, 2, 3, 4, 5, 3, 8, 9],
    "long": [0, 1, 7, 8, 9, 12, 15, 16, 17, 31, 32, 33, 36, 40, 63, 64, 65, 0],      # mean 25
    "below": [17, 18, 18, 18, 18, 18], "mean": [18, 18, 18], "above": [18, 19, 18],
}


@pytest.mark.parametrize("D", [4, 8, 16, 20, 32, 36, 40, 60, 64, 68, 128, 200, 256, 320, 512, 1020])
@pytest.mark.parametrize("name", list(LENGTHS))
def test_pooled_forward(oracle, name, D):
    T, lens = 3, np.tile(np.array(LENGTHS[name], dtype=np.int64), 5)
    B = len(lens)
    wl = W.Workload("pooled", (5, 70, 3000), D=D, B=B, alpha=None)
    rng = np.random.default_rng(D + B)
    off = np.concatenate([[0], np.cumsum(np.concatenate([rng.permutation(lens) for _ in range(T)]))]).astype(np.int32)
    idx = np.concatenate([rng.integers(0, wl.rows[t], off[(t + 1) * B] - off[t * B]) for t in range(T)]).astype(np.int32)
    c = Case(wl, max_lookups=len(idx))
    tables = W.tables_np(wl)
    scales, _ = oracle.scale_refresh(tables, c.row_off, D, c.bits_np)
    for want_codes in (False, True):
        out, codes = c.gpu_fwd(c.dev(tables), idx, off, c.dev(scales), want_codes=want_codes)
        o = oracle.emb_fwd(tables, c.row_off, D, B, idx, off, scales, c.bits_np)
        assert bit_equal(out, o)
    table_of = np.repeat(np.arange(T), [off[(t + 1) * B] - off[t * B] for t in range(T)])
    rows = tables.reshape(-1, D)[c.row_off[table_of] + idx]
    want = np.clip(np.rint(rows / scales[table_of][:, None]), -8, 7).astype(np.int8)      # (4 bits; one FP32 division)
    assert bit_equal(codes, want)
    c.ctx.close()
