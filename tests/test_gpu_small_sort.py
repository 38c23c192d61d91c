"""GPU parity of the block sort of small batches at its edges: around each block size, uneven tables that do not fit
the block, one lookup, one row, many tables."""
import numpy as np
import pytest

from dqrm_inputs import workloads as W
from gpu_util import Case, bit_equal

pytestmark = pytest.mark.gpu

# lookups per table
COUNTS = {
    "around_256": [255, 256, 257, 1], "around_512": [512, 511, 513, 0], "around_1024": [1024, 1023, 1025, 1024],
    "one_table_holds_all": [0, 3, 4000, 0], "single": [1], "many_tables": [2048, 2047, 31, 32, 33] * 16,
}


@pytest.mark.parametrize("rows", [1, 7, 300, 70_000])
@pytest.mark.parametrize("name", list(COUNTS))
def test_block_sort(oracle, name, rows):
    counts = COUNTS[name]
    B, D = max(1, max(counts)), 8
    wl = W.Workload("small", tuple(max(1, rows + t) for t in range(len(counts))), D=D, B=B, alpha=None)
    rng = np.random.default_rng(rows + B)
    idx = np.concatenate([rng.integers(0, wl.rows[t], n) for t, n in enumerate(counts)]).astype(np.int32)
    lens = np.zeros((wl.T, B), dtype=np.int64)
    for t, n in enumerate(counts):                  # some bags empty, some with several indices
        np.add.at(lens[t], rng.integers(0, B, n) if t % 2 else np.arange(n), 1)
    off = np.concatenate([[0], np.cumsum(lens.reshape(-1))]).astype(np.int32)
    go = rng.standard_normal((B, wl.T, D)).astype(np.float32)
    c = Case(wl, max_lookups=len(idx))
    ur, uo, gr = c.gpu_bwd_two_calls(idx, off, go)
    o_ur, o_uo, o_gr = oracle.emb_bwd(go, wl.T, D, B, idx, off)
    assert bit_equal(uo, o_uo) and bit_equal(ur, o_ur)
    # at most 4000 terms of magnitude below 6 in FP64 in two orders, each sum rounded once
    np.testing.assert_allclose(gr, o_gr, rtol=2.0 ** -23, atol=12.0 * 4000 ** 2 * 2.0 ** -53)
    c.ctx.close()


# (lookups per table, bags per table, kernel): small batches in which one table is beyond a block, whose cluster then sorts it
UNEVEN = {
    "shared_1": ([13, 0, 3_000] + [40] * 23, 150, "cluster_sort_kernel"), "shared_2": ([9_000, 500, 1] + [300] * 21, 600, "cluster_sort_kernel"),
    "edges_1": ([511, 512, 513, 514] + [0, 1], 700, "cluster_sort_kernel"), "edges_2": ([1023, 1024, 1025, 90] + [0, 1], 1100, "cluster_sort_kernel"),
    "beyond_the_clusters": ([700] * 98 + [60_000, 1], 800, "cluster_sort_kernel"),
    "edges_4": ([2047, 2048, 2049, 2050] + [1_400] * 60, 2100, "cluster_sort_kernel"),
    # as many lookups as bags, but not one in each
    "in_memory": ([400, 0, 0, 0], 100, "small_sort_kernel"), "in_memory_wide": ([3_000, 1_000, 72, 24], 1_024, "small_sort_kernel"),
}


@pytest.mark.parametrize("rows", [1, 300, 70_000])
@pytest.mark.parametrize("name", list(UNEVEN))
def test_uneven_tables(oracle, name, rows):
    counts, B, kernel = UNEVEN[name]
    D = 8
    wl = W.Workload("uneven", tuple(max(1, rows + t) for t in range(len(counts))), D=D, B=B, alpha=None)
    rng = np.random.default_rng(rows + B)
    idx = np.concatenate([rng.integers(0, wl.rows[t], n) for t, n in enumerate(counts)]).astype(np.int32)
    lens = np.zeros((wl.T, B), dtype=np.int64)
    for t, n in enumerate(counts):
        np.add.at(lens[t], rng.integers(0, B, n), 1)
    off = np.concatenate([[0], np.cumsum(lens.reshape(-1))]).astype(np.int32)
    go = rng.standard_normal((B, wl.T, D)).astype(np.float32)
    c = Case(wl, max_lookups=len(idx))
    c.ctx.profile_begin()
    ur, uo, gr = c.gpu_bwd_two_calls(idx, off, go)
    names = set(c.ctx.profile_end())
    assert names & {"small_sort_kernel", "cluster_sort_kernel", "rs_scatter_kernel"} == {kernel}, names
    o_ur, o_uo, o_gr = oracle.emb_bwd(go, wl.T, D, B, idx, off)
    assert bit_equal(uo, o_uo) and bit_equal(ur, o_ur)
    # at most 60,000 terms of magnitude below 6 in FP64 in two orders, each sum rounded once
    np.testing.assert_allclose(gr, o_gr, rtol=2.0 ** -23, atol=12.0 * max(counts) ** 2 * 2.0 ** -53)
    c.ctx.close()


@pytest.mark.parametrize("rows", [1 << 16, (1 << 16) + 1, 1 << 24, 20_000_000])      # two, three and four digits
@pytest.mark.parametrize("n", [257, 511, 512, 513, 1025, 2047, 2048])
def test_block_radix_sort(oracle, rows, n):
    """The block's radix sort at the edges of its groups and of its digits; rows at both ends of the table, and one that a
    third of the lookups hit."""
    D, T = 4, 2
    wl = W.Workload("radix", (rows, rows), D=D, B=n, alpha=None)
    rng = np.random.default_rng(rows + n)
    idx = rng.integers(0, rows, T * n).astype(np.int32)
    idx[rng.random(T * n) < 0.33] = rows // 3
    idx[[0, 1, n - 1, n, T * n - 1]] = [rows - 1, 0, rows - 1, 0, rows - 1]
    off = np.arange(T * n + 1, dtype=np.int32)
    go = rng.standard_normal((n, T, D)).astype(np.float32)
    c = Case(wl)
    c.ctx.profile_begin()
    ur, uo, gr = c.gpu_bwd_two_calls(idx, off, go)
    assert "small_sort_kernel" in c.ctx.profile_end()
    o_ur, o_uo, o_gr = oracle.emb_bwd(go, T, D, n, idx, off)
    assert bit_equal(uo, o_uo) and bit_equal(ur, o_ur)
    # at most 800 terms of magnitude below 6 in FP64 in two orders, each sum rounded once
    np.testing.assert_allclose(gr, o_gr, rtol=2.0 ** -23, atol=12.0 * 800 ** 2 * 2.0 ** -53)
    c.ctx.close()


@pytest.mark.parametrize("counts,B", [
    ([6_000, 0, 0], 2_000), ([15_000, 17] + [400] * 7 + [2_183], 2_000), ([1] * 25 + [53_223], 2_048), ([2_049] + [1_050] * 35 + [1_901], 1_100),
    ([80, 2_046], 1_063), ([70_000] + [100] * 35 + [2_276], 2_048),
])
@pytest.mark.parametrize("rows", [1, 70_000])
def test_even_batches_that_are_uneven(oracle, rows, counts, B):
    """As many lookups as bags, on average more than a thousand a table, but some or most of them in one."""
    T, D = len(counts), 8
    counts = counts[:-1] + [counts[-1] + T * B - sum(counts)]
    wl = W.Workload("even", tuple(max(1, rows + t) for t in range(T)), D=D, B=B, alpha=None)
    rng = np.random.default_rng(rows + B)
    idx = np.concatenate([rng.integers(0, wl.rows[t], n) for t, n in enumerate(counts)]).astype(np.int32)
    lens = np.zeros((T, B), dtype=np.int64)
    for t, n in enumerate(counts):
        np.add.at(lens[t], rng.integers(0, B, n), 1)
    off = np.concatenate([[0], np.cumsum(lens.reshape(-1))]).astype(np.int32)
    assert len(idx) == T * B
    go = rng.standard_normal((B, T, D)).astype(np.float32)
    c = Case(wl)
    ur, uo, gr = c.gpu_bwd(idx, off, go)
    o_ur, o_uo, o_gr = oracle.emb_bwd(go, T, D, B, idx, off)
    assert bit_equal(uo, o_uo) and bit_equal(ur, o_ur)
    # at most T * B terms of magnitude below 6 in FP64 in two orders, each sum rounded once
    np.testing.assert_allclose(gr, o_gr, rtol=2.0 ** -23, atol=12.0 * max(counts) ** 2 * 2.0 ** -53)
    c.ctx.close()
