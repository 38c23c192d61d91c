"""GPU parity of the forward and the packed lookup in both orders of their blocks, with more bags than one pass of a table's
blocks takes: on both sides of the mean bag lengths and widths at which the order changes."""
import numpy as np
import pytest

from dqrm_inputs import workloads as W
from gpu_util import Case, bit_equal

pytestmark = pytest.mark.gpu


# features, bags, mean indices a bag
@pytest.mark.parametrize("D,B,bag", [
    (4, 30_500, 1), (64, 30_500, 1), (4, 30_500, 2), (16, 8_000, 2), (32, 4_000, 2), (32, 4_000, 15), (32, 4_000, 16), (48, 2_000, 4), (64, 2_000, 4),
    (64, 2_000, 5), (128, 1_000, 2), (128, 1_000, 3), (200, 1_000, 2),
])
def test_order_of_the_blocks(oracle, D, B, bag):
    import torch

    T = 40                               # 119 blocks a table
    wl = W.Workload("order", tuple(3 + 20 * t for t in range(T)), D=D, B=B, alpha=None)
    rng = np.random.default_rng(D + bag)
    lens = np.full(T * B, bag, dtype=np.int64)
    if bag > 1:                          # uneven, of the same mean
        half = rng.permutation(T * B)[:T * B // 2 * 2]
        lens[half[::2]] -= 1
        lens[half[1::2]] += 1
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    table = np.repeat(np.arange(T), lens.reshape(T, B).sum(1))
    idx = (rng.random(off[-1]) * np.array(wl.rows)[table]).astype(np.int32)
    c = Case(wl, max_lookups=len(idx))
    tables = W.tables_np(wl)
    scales, _ = oracle.scale_refresh(tables, c.row_off, D, c.bits_np)
    want = oracle.emb_fwd(tables, c.row_off, D, B, idx, off, scales, c.bits_np)
    d_tables, d_scales = c.dev(tables), c.dev(scales)
    out, _ = c.gpu_fwd(d_tables, idx, off, d_scales, want_codes=False)
    assert bit_equal(out, want)
    if bag == 2:
        out, _ = c.gpu_fwd(d_tables, idx, off, d_scales, want_codes=True)
        assert bit_equal(out, want)
    packed, d_out = c.empty(c.ctx.packed_bytes(wl.bits), torch.uint8), c.empty((B, T, D), torch.float32)
    c.ctx.pack_tables(d_tables, d_scales, wl.bits, packed)
    c.ctx.packed_fwd(packed, c.dev(idx), c.dev(off), d_scales, wl.bits, d_out, B=B, L=len(idx))
    c.ctx.raise_on_device_error()
    assert bit_equal(d_out.cpu().numpy(), want)
    c.ctx.close()


# one-index batches of few warps, which take 32 bags each (from twelve warps an SM of 148 on: 26 tables of 2177) down to one step of
# rows: whole and cut warps, and bags of none and of two
@pytest.mark.parametrize("D", [16, 20, 32, 36, 64, 100, 128, 200, 256, 1020])
@pytest.mark.parametrize("T,B", [(1, 1), (3, 5), (2, 33), (5, 100), (26, 517), (7, 2049), (26, 2048), (26, 2176), (26, 2177)])
def test_few_warps(oracle, D, T, B):
    if T * B > 20_000 and D not in (32, 64, 100, 256):
        pytest.skip("the larger batches take one width of each kind")
    wl = W.Workload("few", tuple(3 + 50 * t for t in range(T)), D=D, B=B, alpha=None)
    rng = np.random.default_rng(D + B)
    lens = np.ones(T * B, dtype=np.int64)
    for odd in (False, True):
        if odd:                          # (as many lookups as bags all the same)
            if T * B < 5:
                break
            at = rng.permutation(T * B)[:T * B // 50 * 2 + 2]
            lens[at[::2]], lens[at[1::2]] = 0, 2
        off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
        table = np.repeat(np.arange(T), lens.reshape(T, B).sum(1))
        idx = (rng.random(off[-1]) * np.array(wl.rows)[table]).astype(np.int32)
        c = Case(wl, max_lookups=len(idx))
        tables = W.tables_np(wl)
        scales, _ = oracle.scale_refresh(tables, c.row_off, D, c.bits_np)
        out, _ = c.gpu_fwd(c.dev(tables), idx, off, c.dev(scales), want_codes=False)
        assert bit_equal(out, oracle.emb_fwd(tables, c.row_off, D, B, idx, off, scales, c.bits_np))
        c.ctx.close()
