"""GPU parity of the small batch's step in one launch behind the forward, at its edges: tables of no, one and many
lookups, runs that cross many lane groups' shares, an uneven batch whose table does not fit the block, feature sizes
whose last lanes are idle, and the batch on either side of the largest that it takes."""
import numpy as np
import pytest

from dqrm_inputs import workloads as W
from gpu_util import Case, bit_equal

pytestmark = pytest.mark.gpu

# feature size: lookups per table
SHAPES = {
    "single": (16, [1]), "empty_tables": (4, [0, 3, 0, 0, 40, 0]), "tiny": (16, [128, 128, 128, 128]), "idle_lanes": (20, [33, 257, 64]),
    "block": (16, [512, 511, 513, 512]), "beyond_it": (16, [513, 513, 513, 513]), "all": (32, [512] * 8), "and_one": (4, [512] * 7 + [513]),
    "one_table_holds_all": (8, [0, 2, 3200, 0, 0, 0, 1, 0]), "wide": (128, [127, 128]), "narrow": (4, [300] * 13),
    "many_tables": (8, [1, 0, 40, 33] * 30),
    # uneven batches up to the most that one block may have to take alone, and one lookup beyond
    "one_block_takes_most": (16, [3, 0, 1500, 33]), "and_one_more": (16, [3, 0, 1501, 33]), "few_in_many_tables": (8, [1, 0, 10, 13] * 30),
    "widest_uneven": (64, [500, 1, 11]), "too_wide_uneven": (64, [501, 1, 11]),
}


@pytest.mark.parametrize("rows", [1, 9, 50_000])
@pytest.mark.parametrize("name", list(SHAPES))
def test_small_step(oracle, name, rows):
    import torch

    D, counts = SHAPES[name]
    T, B = len(counts), max(1, max(counts))
    wl = W.Workload("step", tuple(rows + t for t in range(T)), D=D, B=B, alpha=None)
    rng = np.random.default_rng(rows + B + D)
    idx = np.concatenate([rng.integers(0, wl.rows[t], n) for t, n in enumerate(counts)]).astype(np.int32)
    lens = np.zeros((T, B), dtype=np.int64)
    for t, n in enumerate(counts):
        np.add.at(lens[t], rng.integers(0, B, n) if t % 2 else np.arange(n), 1)
    off = np.concatenate([[0], np.cumsum(lens.reshape(-1))]).astype(np.int32)
    # gradients are multiples of 2^-8 below 4, so sums of a few thousand are exact in FP32 and every output has one value
    go = (rng.integers(-1024, 1025, (B, T, D)) / 256).astype(np.float32)
    L = len(idx)
    c = Case(wl, max_lookups=L)
    o_tables = W.tables_np(wl)
    o_scales, _ = oracle.scale_refresh(o_tables, c.row_off, D, c.bits_np)
    d_tables = c.dev(o_tables)
    r = oracle.train_step(o_tables, c.row_off, D, B, idx, off, go, o_scales, c.bits_np, wl.lr)
    out, uo, gs = c.empty((B, T, D), torch.float32), c.empty(T + 1, torch.int32), c.empty(T, torch.float32)
    ur, gr, codes = c.empty(L, torch.int32), c.empty((L, D), torch.float32), c.empty((L, D), torch.int8)
    c.ctx.train_step(d_tables, c.dev(idx), c.dev(off), c.dev(go), c.dev(o_scales), c.bits, out, ur, uo, gr, codes, gs,
                     wl.lr, B=B, L=L)
    c.ctx.raise_on_device_error()
    U = int(r["uniq_off"][-1])
    np.testing.assert_allclose(out.cpu().numpy(), r["out"], rtol=1e-5, atol=1e-6)      # (the forward's own tolerance)
    assert bit_equal(uo.cpu().numpy(), r["uniq_off"]) and bit_equal(ur.cpu().numpy()[:U], r["unique_rows"])
    assert bit_equal(gr.cpu().numpy()[:U], r["grad_rows"]) and bit_equal(gs.cpu().numpy(), r["grad_scales"])
    assert bit_equal(codes.cpu().numpy()[:U], r["codes"]) and bit_equal(d_tables.cpu().numpy(), o_tables)
    c.ctx.close()


@pytest.mark.parametrize("boundary", [(0, 1), (2, 500), (2, -3), (4, 80)])
def test_unusable_boundaries_touch_no_row(boundary):
    import torch
    import paper_2410_20046_b200 as dq

    T, B, D = 4, 32, 16
    wl = W.Workload("step", (40,) * T, D=D, B=B, alpha=None)
    c = Case(wl)
    tables = W.tables_np(wl)
    d_tables = c.dev(tables)
    off = np.arange(T * B + 1, dtype=np.int32)
    off[boundary[0] * B] = boundary[1]
    out, uo, gs = c.empty((B, T, D), torch.float32), c.empty(T + 1, torch.int32), c.empty(T, torch.float32)
    ur, gr = c.empty(T * B, torch.int32), c.empty((T * B, D), torch.float32)
    c.ctx.train_step(d_tables, c.dev(np.zeros(T * B, np.int32)), c.dev(off), c.dev(np.ones((B, T, D), np.float32)),
                     c.dev(np.full(T, 0.1, np.float32)), c.bits, out, ur, uo, gr, c.empty((T * B, D), torch.int8), gs, wl.lr,
                     B=B, L=T * B)
    with pytest.raises(dq.DqrmError):
        c.ctx.raise_on_device_error()
    assert bit_equal(d_tables.cpu().numpy(), tables)
    c.ctx.close()


def test_contexts_of_many_and_of_few_tables_take_turns(oracle):
    """Two live contexts on one device: the kernel's shared-memory limit is the device's, not a context's."""
    import torch

    B, D = 16, 16
    cases = []
    for T in (100, 3):
        wl = W.Workload("turns", (40,) * T, D=D, B=B, alpha=None)
        c = Case(wl)
        o_tables = W.tables_np(wl)
        o_scales, _ = oracle.scale_refresh(o_tables, c.row_off, D, c.bits_np)
        cases.append((c, o_tables, o_scales, c.dev(o_tables)))
    for turn in range(3):
        for c, o_tables, o_scales, d_tables in cases:
            wl, L = c.wl, c.wl.T * B
            rng = np.random.default_rng(turn + wl.T)
            idx = rng.integers(0, 40, L).astype(np.int32)
            off = np.arange(L + 1, dtype=np.int32)
            go = (rng.integers(-1024, 1025, (B, wl.T, D)) / 256).astype(np.float32)
            r = oracle.train_step(o_tables, c.row_off, D, B, idx, off, go, o_scales, c.bits_np, wl.lr)
            out, uo, gs = c.empty((B, wl.T, D), torch.float32), c.empty(wl.T + 1, torch.int32), c.empty(wl.T, torch.float32)
            ur, gr, codes = c.empty(L, torch.int32), c.empty((L, D), torch.float32), c.empty((L, D), torch.int8)
            c.ctx.train_step(d_tables, c.dev(idx), c.dev(off), c.dev(go), c.dev(o_scales), c.bits, out, ur, uo, gr, codes,
                             gs, wl.lr, B=B, L=L)
            c.ctx.raise_on_device_error()
            U = int(r["uniq_off"][-1])
            assert bit_equal(uo.cpu().numpy(), r["uniq_off"]) and bit_equal(codes.cpu().numpy()[:U], r["codes"])
            assert bit_equal(d_tables.cpu().numpy(), o_tables)
    for c, *_ in cases:
        c.ctx.close()


# the backward alone: feature size, lookups per table, launches: one up to the line, two (sort and sum) beyond it.  An index a bag:
ALONE_EVEN = {
    "single": (16, [1], 1), "tiny": (16, [128] * 4, 1), "most_lookups": (16, [225] * 16, 1), "a_table_more": (16, [225] * 17, 2),
    "most_values": (32, [256] * 8, 1), "a_table_of_values_more": (32, [256] * 9, 2), "most_of_a_table": (32, [512] * 2, 1),
    "a_table_too_long": (16, [513] * 2, 2), "a_table_too_wide": (64, [257] * 2, 2), "narrow": (4, [384] * 2, 1), "too_narrow": (4, [385] * 2, 2),
    "many_tables": (16, [64] * 32, 1), "one_too_many": (16, [64] * 33, 2), "idle_lanes": (20, [90] * 7, 1), "wide": (128, [128] * 4, 1),
}
# and others:
ALONE_UNEVEN = {
    "empty_tables": (4, [0, 3, 0, 0, 40, 0], 1), "one_holds_most": (16, [3, 0, 1064, 33], 1), "and_one_more": (16, [3, 0, 1065, 33], 2),
    "widest": (64, [500, 1, 11], 1), "too_wide": (64, [501, 1, 11], 2), "idle_lanes": (20, [33, 934, 57], 1), "idle_lanes_more": (20, [33, 935, 57], 2),
    "many_tables": (8, [1, 0, 7, 13] * 30, 1), "in_memory": (8, [0, 2, 900, 1], 1),
}


@pytest.mark.parametrize("rows", [1, 9, 50_000])
@pytest.mark.parametrize("name", list(ALONE_EVEN) + ["uneven " + k for k in ALONE_UNEVEN])
def test_small_backward(oracle, name, rows):
    """The backward alone in one launch, on both sides of what it takes; what the profile names is what runs."""
    even = not name.startswith("uneven ")
    D, counts, launches = ALONE_EVEN[name] if even else ALONE_UNEVEN[name[7:]]
    T, B = len(counts), counts[0] if even else max(counts)
    wl = W.Workload("bwd", tuple(rows + t for t in range(T)), D=D, B=B, alpha=None)
    rng = np.random.default_rng(rows + B + D)
    idx = np.concatenate([rng.integers(0, wl.rows[t], n) for t, n in enumerate(counts)]).astype(np.int32)
    lens = np.ones((T, B), dtype=np.int64)
    if not even:
        lens[:] = 0
        for t, n in enumerate(counts):
            np.add.at(lens[t], rng.integers(0, B, n) if t % 2 else np.arange(n), 1)
    off = np.concatenate([[0], np.cumsum(lens.reshape(-1))]).astype(np.int32)
    assert len(idx) == off[-1] and (len(idx) == T * B) == even
    go = (rng.integers(-1024, 1025, (B, T, D)) / 256).astype(np.float32)      # (exact sums, as above)
    c = Case(wl, max_lookups=len(idx))
    before = c.ctx.launch_count()
    got, want = c.gpu_bwd(idx, off, go), oracle.emb_bwd(go, T, D, B, idx, off)
    assert c.ctx.launch_count() - before == launches
    c.ctx.profile_begin()
    again = c.gpu_bwd(idx, off, go)
    named = c.ctx.profile_end()
    assert sum(n for _, n in named.values()) == launches and ("small_step_kernel" in named) == (launches == 1), named
    for g, a, w in zip(got, again, want[:3]):
        assert bit_equal(g, w) and bit_equal(a, w)
    c.ctx.close()
