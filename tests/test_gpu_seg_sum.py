"""GPU parity of the segmented sum at the sizes where its split can go wrong: tables whose runs end on, before and
behind the edges of tiles and of the warps' ranges, a run that covers many ranges, one lookup, every row width class."""
import numpy as np
import pytest

from dqrm_inputs import workloads as W
from gpu_util import Case, bit_equal

pytestmark = pytest.mark.gpu

# lengths of the runs of equal rows, table by table (rows 0, 1, 2, ...)
SPLITS = {
    "one": [[1], [1]],
    "tile_edges": [[31, 1, 1, 31, 32, 33, 63, 1, 64, 65, 31], [32], [64], [1, 63, 128, 7]],
    "all_unique": [[1] * 700, [1] * 70, [2] * 99],
    "one_run_over_ranges": [[3, 240_000, 5], [1]],
    "long_and_short": [[1, 20_000] * 6 + [1] * 3_000, [150_000]],
}


@pytest.mark.parametrize("sort_path", [0, 1])
@pytest.mark.parametrize("D", [4, 8, 12, 16, 20, 32, 36, 64, 128, 200])
@pytest.mark.parametrize("split", list(SPLITS))
def test_runs_at_the_edges(oracle, split, D, sort_path):
    if split in ("one_run_over_ranges", "long_and_short") and D not in (4, 16, 20, 64, 200):
        pytest.skip("the large splits take one size of each kind")
    runs = SPLITS[split]
    counts = [sum(r) for r in runs]
    B = max(counts)                     # bags of one index; tables with fewer lookups end in empty bags
    wl = W.Workload("runs", tuple(max(4, len(r)) for r in runs), D=D, B=B, alpha=None)
    rng = np.random.default_rng(len(split) + D)
    idx = np.concatenate([rng.permutation(np.repeat(np.arange(len(r)), r)) for r in runs]).astype(np.int32)
    lens = np.zeros((wl.T, B), dtype=np.int64)
    for t, n in enumerate(counts):
        lens[t, :n] = 1
    off = np.concatenate([[0], np.cumsum(lens.reshape(-1))]).astype(np.int32)
    go = rng.standard_normal((B, wl.T, D)).astype(np.float32)
    c = Case(wl, max_lookups=len(idx))
    c.ctx.set_sort_path(sort_path)
    ur, uo, gr = c.gpu_bwd(idx, off, go)
    o_ur, o_uo, o_gr = oracle.emb_bwd(go, wl.T, D, B, idx, off)
    assert bit_equal(uo, o_uo) and bit_equal(ur, o_ur)
    # n terms of magnitude below 6 in FP64, in two orders: the sums differ by at most 2 n^2 * 6 * 2^-53 and each is
    # rounded once, to within 2^-24 of itself
    n = max(max(r) for r in runs)
    np.testing.assert_allclose(gr, o_gr, rtol=2.0 ** -23, atol=12.0 * n * n * 2.0 ** -53)
    c.ctx.close()


# tables of 1,024 to 98,304 lookups on average, which the clusters sort and number themselves: a run over hundreds of
# ranges in a table alone (sixteen blocks) and beside small ones (eight), a table beyond its blocks' shared memory, runs
# on the edges of tiles
CLUSTER_SPLITS = {
    "one_run": [[3, 80_000, 5]],
    "one_run_uneven": [[7, 1]] * 2 + [[3, 40_000, 5]] + [[1, 31, 32, 33] * 20, [1] * 2_500, [64] * 33, [2, 30] * 40],
    "edges": [[31, 1, 1, 31, 32, 33, 63, 1, 64, 65, 31] * 9] * 7,
}


@pytest.mark.parametrize("D", [8, 16, 32, 64, 100, 128, 200, 256, 1020, 1024])
@pytest.mark.parametrize("split", list(CLUSTER_SPLITS))
def test_runs_of_the_cluster_sort(oracle, split, D):
    if D > 128 and split == "one_run":
        pytest.skip("the table alone takes the narrower rows")
    runs = CLUSTER_SPLITS[split]
    counts = [sum(r) for r in runs]
    B = max(counts)                     # bags of one index; tables with fewer lookups end in empty bags
    wl = W.Workload("runs", tuple(max(4, len(r)) for r in runs), D=D, B=B, alpha=None)
    rng = np.random.default_rng(len(split) + D)
    idx = np.concatenate([rng.permutation(np.repeat(np.arange(len(r)), r)) for r in runs]).astype(np.int32)
    lens = np.zeros((wl.T, B), dtype=np.int64)
    for t, n in enumerate(counts):
        lens[t, :n] = 1
    off = np.concatenate([[0], np.cumsum(lens.reshape(-1))]).astype(np.int32)
    L = len(idx)
    # of the bags behind the last lookup nothing is read: one row of zeros would do, so only the used ones are drawn
    go = np.zeros((B, wl.T, D), dtype=np.float32)
    for t, n in enumerate(counts):
        go[:n, t] = rng.standard_normal((n, D), dtype=np.float32)
    c = Case(wl, max_lookups=L)
    c.ctx.profile_begin()
    ur, uo, gr = c.gpu_bwd(idx, off, go)
    names = set(c.ctx.profile_end())
    assert names & {"small_sort_kernel", "cluster_sort_kernel", "rs_scatter_kernel"} == {"cluster_sort_kernel"}, names
    o_ur, o_uo, o_gr = oracle.emb_bwd(go, wl.T, D, B, idx, off)
    assert bit_equal(uo, o_uo) and bit_equal(ur, o_ur)
    # as above
    n = max(max(r) for r in runs)
    np.testing.assert_allclose(gr, o_gr, rtol=2.0 ** -23, atol=12.0 * n * n * 2.0 ** -53)
    c.ctx.close()


@pytest.mark.parametrize("D", [4, 8, 16, 20, 32, 36, 48])
@pytest.mark.parametrize("n", [1, 7, 8, 9, 255, 257, 4_099])
def test_runs_of_lane_groups(oracle, n, D):
    """Rows that take a lane group, where the groups' ranges, the tables and the runs all end at different entries: tables
    of one lookup beside larger ones, runs of one to nine entries, signed zeros among the gradients."""
    rng = np.random.default_rng(n + D)
    counts = [n, 1, 0, max(1, n // 3), 5]
    B = max(counts)
    runs = [np.repeat(np.arange(c), rng.integers(1, 10, c))[:c] for c in counts]
    wl = W.Workload("groups", tuple(max(4, c) for c in counts), D=D, B=B, alpha=None)
    idx = np.concatenate([rng.permutation(r) for r in runs]).astype(np.int32)
    lens = np.zeros((wl.T, B), dtype=np.int64)
    for t, c in enumerate(counts):
        lens[t, :c] = 1
    off = np.concatenate([[0], np.cumsum(lens.reshape(-1))]).astype(np.int32)
    go = rng.standard_normal((B, wl.T, D)).astype(np.float32)
    go[rng.random(go.shape) < 0.1] = -0.0
    c = Case(wl, max_lookups=len(idx))
    ur, uo, gr = c.gpu_bwd_two_calls(idx, off, go)
    o_ur, o_uo, o_gr = oracle.emb_bwd(go, wl.T, D, B, idx, off)
    assert bit_equal(uo, o_uo) and bit_equal(ur, o_ur)
    # nine terms of magnitude below 6 in FP64 in two orders, each sum rounded once
    np.testing.assert_allclose(gr, o_gr, rtol=2.0 ** -23, atol=12.0 * 9 * 9 * 2.0 ** -53)
    c.ctx.close()


@pytest.mark.parametrize("rows", [1, 2, 3, 5, 1 << 10, (1 << 10) + 1, 1 << 20, (1 << 20) + 1])      # one to three digits of one bit and up
def test_radix_sort_digits(oracle, rows):
    """The radix sort's ranks and places at the edges of its digits and of its tiles of 4096: bags of zero to five, a
    row that a third of the lookups hit, rows at both ends of the table."""
    rng = np.random.default_rng(rows)
    T, B, D = 3, 4_100, 4
    wl = W.Workload("digits", (rows, rows, max(1, rows // 2)), D=D, B=B, alpha=None)
    lens = rng.integers(0, 6, T * B)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    table = np.repeat(np.arange(T), lens.reshape(T, B).sum(1))
    idx = (rng.random(off[-1]) * np.array(wl.rows)[table]).astype(np.int32)
    idx[rng.random(len(idx)) < 0.33] = wl.rows[2] // 3
    idx[0], idx[-1] = rows - 1, wl.rows[2] - 1
    go = rng.standard_normal((B, T, D)).astype(np.float32)
    c = Case(wl, max_lookups=len(idx))
    c.ctx.set_sort_path(1)
    ur, uo, gr = c.gpu_bwd(idx, off, go)
    o_ur, o_uo, o_gr = oracle.emb_bwd(go, T, D, B, idx, off)
    assert bit_equal(uo, o_uo) and bit_equal(ur, o_ur)
    # at most 25,000 terms of magnitude below 6 in FP64 in two orders, each sum rounded once
    np.testing.assert_allclose(gr, o_gr, rtol=2.0 ** -23, atol=12.0 * 25_000 ** 2 * 2.0 ** -53)
    c.ctx.close()


# On 148 SMs a lane group's range is one round of eight entries up to 47 K lookups of 36 to 48 features, 95 K of 20 to 32, 189 K of
# 12 and 16, 379 K of 8 and 758 K of 4: these take more rounds
@pytest.mark.parametrize("D,B", [(36, 7_001), (48, 12_003), (44, 40_001), (20, 14_002), (32, 27_001), (24, 60_005), (12, 30_003), (16, 50_001), (8, 60_001), (4, 120_003)])
@pytest.mark.parametrize("sort_path", [0, 1])
def test_lane_groups_of_many_rounds(oracle, D, B, sort_path):
    rng = np.random.default_rng(D)
    rows = (40_000, 3, 900_000, 1)
    T = len(rows)
    wl = W.Workload("rounds", rows, D=D, B=B, alpha=None)
    lens = rng.integers(0, 6, T * B)
    lens[:B // 3] = 0                               # a table of fewer lookups
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    L = int(off[-1])
    table = np.repeat(np.arange(T), lens.reshape(T, B).sum(1))
    idx = (rng.random(L) ** rng.choice([1, 8], L) * np.array(rows)[table]).astype(np.int32)      # runs of one to thousands
    assert L > 8 * 2960 * (32 // (1 if D <= 4 else 2 if D <= 8 else 4 if D <= 16 else 8 if D <= 32 else 16))
    go = rng.standard_normal((B, T, D), dtype=np.float32)
    c = Case(wl, max_lookups=L)
    c.ctx.set_sort_path(sort_path)
    ur, uo, gr = c.gpu_bwd(idx, off, go)
    o_ur, o_uo, o_gr = oracle.emb_bwd(go, T, D, B, idx, off)
    assert bit_equal(uo, o_uo) and bit_equal(ur, o_ur)
    # n terms of magnitude below 6 in FP64 in two orders, each sum rounded once
    n = int(np.bincount(idx + 1_000_000 * table).max())
    np.testing.assert_allclose(gr, o_gr, rtol=2.0 ** -23, atol=12.0 * n * n * 2.0 ** -53)
    c.ctx.close()


@pytest.mark.parametrize("D", [8, 64])
@pytest.mark.parametrize("rows", [1, 3, 257, 70_001, 3_000_000])
@pytest.mark.parametrize("where", ["all", "first", "last", "ends", "one"])
def test_table_alone_by_its_parts(oracle, where, rows, D):
    """A large table alone, whose rows four clusters share: lookups over all of them, in the first or the last share only (the
    other lists stay empty), on the shares' edges, in one row; an index a bag and uneven bags."""
    rng = np.random.default_rng(rows + D)
    edges = sorted({min(max(rows * q // 4 + d, 0), rows - 1) for q in range(5) for d in (-1, 0, 1)})
    for bags in (False, True):
        B = 17_001 if not bags else 9_000
        lens = rng.integers(0, 5, B) if bags else np.ones(B, dtype=np.int64)
        L = int(lens.sum())
        assert 16 * 1024 <= L
        u = rng.random(L)
        idx = {"all": u * rows, "first": u * max(1, rows // 4), "last": rows - 1 - u * max(1, rows // 4),
               "ends": np.array(edges)[(u * len(edges)).astype(int)], "one": np.full(L, rows // 2)}[where].astype(np.int32).clip(0, rows - 1)
        off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
        go = rng.standard_normal((B, 1, D)).astype(np.float32)
        c = Case(W.Workload("alone", (rows,), D=D, B=B, alpha=None), max_lookups=L)
        ur, uo, gr = c.gpu_bwd(idx, off, go)
        o_ur, o_uo, o_gr = oracle.emb_bwd(go, 1, D, B, idx, off)
        assert bit_equal(uo, o_uo) and bit_equal(ur, o_ur)
        # n terms of magnitude below 6 in FP64 in two orders, each sum rounded once
        n = int(np.unique(idx, return_counts=True)[1].max())
        np.testing.assert_allclose(gr, o_gr, rtol=2.0 ** -23, atol=12.0 * n * n * 2.0 ** -53)
        c.ctx.close()


# rows of a table alone in which its lookups fall unevenly: four clusters share them at the quantiles of a sample
UNEVEN = {
    "low": lambda rng, R, n: rng.integers(0, max(1, R // 4), n),
    "by_frequency": lambda rng, R, n: np.minimum(R ** rng.random(n), R - 1),
    "padding": lambda rng, R, n: np.where(rng.random(n) < 0.9, 0, rng.integers(0, R, n)),
    "two_rows": lambda rng, R, n: np.where(rng.random(n) < 0.5, R - 1, R // 2),
    "last": lambda rng, R, n: np.full(n, R - 1),
    "beyond": lambda rng, R, n: np.where(rng.random(n) < 0.7, R - 1 - rng.integers(0, max(1, R // 100), n), rng.integers(0, R, n)),
}


@pytest.mark.parametrize("rows", [1, 2, 3, 5, 1_000, 60_000, 70_000, 3_000_000])
@pytest.mark.parametrize("fall", list(UNEVEN))
def test_table_alone_by_quantiles(oracle, fall, rows):
    rng = np.random.default_rng(rows)
    D = 12
    for B, most in ((50_001, 1), (20_003, 6), (33_000, 1)):
        lens = rng.integers(0, most, B) if most > 1 else np.ones(B, dtype=np.int64)
        L = int(lens.sum())
        idx = UNEVEN[fall](rng, rows, L).astype(np.int32)
        off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
        go = rng.standard_normal((B, 1, D)).astype(np.float32)
        c = Case(W.Workload("alone", (rows,), D=D, B=B, alpha=None), max_lookups=L)
        ur, uo, gr = c.gpu_bwd(idx, off, go)
        o_ur, o_uo, o_gr = oracle.emb_bwd(go, 1, D, B, idx, off)
        assert bit_equal(uo, o_uo) and bit_equal(ur, o_ur)
        # n terms of magnitude below 6 in FP64 in two orders, each sum rounded once
        n = int(np.unique(idx, return_counts=True)[1].max())
        np.testing.assert_allclose(gr, o_gr, rtol=2.0 ** -23, atol=12.0 * n * n * 2.0 ** -53)
        c.ctx.close()


def test_low_rows_of_a_table_alone_are_no_slower():
    """Lookups that all fall in the first quarter of the rows: 1.05 times the time of uniform ones (1.37 with even shares)."""
    import torch
    import paper_2410_20046_b200 as dq

    rows, D, L = 4_000_000, 16, 65_536
    ctx = dq.Context([0, rows], D, L, L)
    off = torch.arange(L + 1, dtype=torch.int32, device="cuda")
    go = torch.randn((L, 1, D), device="cuda")
    ur, uo = torch.empty(L, dtype=torch.int32, device="cuda"), torch.empty(2, dtype=torch.int32, device="cuda")
    gr = torch.empty((L, D), device="cuda")
    idx = {high: torch.randint(0, high, (L,), dtype=torch.int32, device="cuda") for high in (rows, rows // 4)}
    times = {high: [] for high in idx}
    for k in range(12):
        for high in idx:
            begin, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            begin.record()
            for _ in range(50):
                ctx.emb_bwd(go, idx[high], off, ur, uo, gr, B=L, L=L)
            end.record()
            torch.cuda.synchronize()
            times[high].append(begin.elapsed_time(end))
    assert np.median(times[rows // 4]) < 1.2 * np.median(times[rows]), times
    ctx.close()


# few tables of 5 K lookups and more, of rows of two and of three digits, which clusters of sixteen and of eight blocks sort
@pytest.mark.parametrize("T,per_table", [(1, 8_191), (1, 8_192), (1, 12_001), (2, 5_119), (2, 5_120), (4, 7_003)])
@pytest.mark.parametrize("rows", [60_000, 70_000])
def test_wide_clusters(oracle, T, per_table, rows):
    rng = np.random.default_rng(T + per_table)
    D, B = 12, per_table
    for bags in (False, True):
        lens = rng.integers(0, 3, T * B) if bags else np.ones(T * B, dtype=np.int64)
        off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
        idx = (rng.random(off[-1]) ** rng.choice([1, 6], off[-1]) * rows).astype(np.int32)
        go = rng.standard_normal((B, T, D), dtype=np.float32)
        c = Case(W.Workload("wide", (rows,) * T, D=D, B=B, alpha=None), max_lookups=len(idx))
        ur, uo, gr = c.gpu_bwd(idx, off, go)
        o_ur, o_uo, o_gr = oracle.emb_bwd(go, T, D, B, idx, off)
        assert bit_equal(uo, o_uo) and bit_equal(ur, o_ur)
        # n terms of magnitude below 6 in FP64 in two orders, each sum rounded once
        n = int(np.bincount(idx + rows * np.repeat(np.arange(T), lens.reshape(T, B).sum(1))).max())
        np.testing.assert_allclose(gr, o_gr, rtol=2.0 ** -23, atol=12.0 * n * n * 2.0 ** -53)
        c.ctx.close()


# many tables, which four blocks or half of a cluster's sort: on both sides of the numbers of tables and lookups at which they do
@pytest.mark.parametrize("D", [8, 36])
@pytest.mark.parametrize("T,per_table", [(18, 2_100), (19, 2_100), (19, 8_192), (19, 8_200), (37, 2_561), (38, 2_600), (38, 9_000), (40, 16_384),
                                         (33, 2_100), (34, 2_100), (34, 8_193), (59, 4_096), (59, 4_097), (66, 4_096), (67, 4_097)])
def test_narrow_clusters(oracle, T, per_table, D):
    if per_table > 9_000 and D > 8:
        pytest.skip("the largest batch takes the narrow rows")
    rng = np.random.default_rng(T + per_table)
    rows = tuple(int(r) for r in rng.choice([1, 3, 300, 70_000], T))
    B = per_table
    for bags in (False, True):
        lens = np.ones((T, B), dtype=np.int64)
        if bags:                         # uneven tables and bags, of the same mean
            half = rng.permutation(T * B)[:T * B // 2 * 2]
            lens.reshape(-1)[half[::2]] -= 1
            lens.reshape(-1)[half[1::2]] += 1
            lens[0, 0] += 1              # (not as many lookups as bags)
        off = np.concatenate([[0], np.cumsum(lens.reshape(-1))]).astype(np.int32)
        table = np.repeat(np.arange(T), lens.sum(1))
        idx = (rng.random(off[-1]) ** rng.choice([1, 6], off[-1]) * np.array(rows)[table]).astype(np.int32)
        go = rng.standard_normal((B, T, D), dtype=np.float32)
        c = Case(W.Workload("narrow", rows, D=D, B=B, alpha=None), max_lookups=len(idx))
        ur, uo, gr = c.gpu_bwd(idx, off, go)
        o_ur, o_uo, o_gr = oracle.emb_bwd(go, T, D, B, idx, off)
        assert bit_equal(uo, o_uo) and bit_equal(ur, o_ur)
        # n terms of magnitude below 6 in FP64 in two orders, each sum rounded once
        n = int(np.bincount(idx + 100_000 * table).max())
        np.testing.assert_allclose(gr, o_gr, rtol=2.0 ** -23, atol=12.0 * n * n * 2.0 ** -53)
        c.ctx.close()


# clusters of four blocks (as many lookups as bags) and clusters of eight of which half works: a table that fits four blocks' shared memory
# to the last pair (3200 at a mean of 2500 lookups a table), one pair more, the last pair that eight blocks hold, and beyond; in
# tables of both halves
@pytest.mark.parametrize("even", [True, False])
@pytest.mark.parametrize("T", [34, 40, 66])
@pytest.mark.parametrize("large", [3_199, 3_200, 3_201, 6_400, 6_401, 40_000])
def test_tables_beyond_half_a_cluster(oracle, T, large, even):
    rng = np.random.default_rng(T + large)
    D, B = 8, 2_500
    counts = np.full(T, (T * B - 2 * large) // (T - 2))
    counts[[2, T - 1]] = large
    counts[0] += T * B - counts.sum() - (not even)
    rows = tuple(int(r) for r in rng.choice([1, 300, 70_000], T))
    lens = np.zeros((T, B), dtype=np.int64)
    for t, n in enumerate(counts):
        np.add.at(lens[t], rng.integers(0, B, n), 1)
    off = np.concatenate([[0], np.cumsum(lens.reshape(-1))]).astype(np.int32)
    table = np.repeat(np.arange(T), counts)
    idx = (rng.random(off[-1]) * np.array(rows)[table]).astype(np.int32)
    go = rng.standard_normal((B, T, D), dtype=np.float32)
    c = Case(W.Workload("half", rows, D=D, B=B, alpha=None), max_lookups=len(idx))
    ur, uo, gr = c.gpu_bwd(idx, off, go)
    o_ur, o_uo, o_gr = oracle.emb_bwd(go, T, D, B, idx, off)
    assert bit_equal(uo, o_uo) and bit_equal(ur, o_ur)
    # n terms of magnitude below 6 in FP64 in two orders, each sum rounded once
    n = int(np.bincount(idx + 100_000 * table).max())
    np.testing.assert_allclose(gr, o_gr, rtol=2.0 ** -23, atol=12.0 * n * n * 2.0 ** -53)
    c.ctx.close()


# hundreds of entries for each of the 4736 warps that 148 SMs hold: one range for each of them, and from 512 on (64 features in long bags;
# 576) ranges of 256 (of 384), several of them for a warp's place
@pytest.mark.parametrize("D,most", [(52, 36), (64, 36), (64, 46), (52, 51), (52, 64)])
@pytest.mark.parametrize("sort_path", [0, 1])
def test_ranges_beyond_the_resident_warps(oracle, D, most, sort_path):
    rng = np.random.default_rng(D)
    rows, B = (40_000, 3, 900_000), 40_003
    T = len(rows)
    wl = W.Workload("ranges", rows, D=D, B=B, alpha=None)
    lens = rng.integers(0, most, T * B)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    L = int(off[-1])
    tiles = {36: 13, 46: 17, 51: 19, 64: 24}[most]
    assert -(-L // (32 * 4736)) >= tiles
    table = np.repeat(np.arange(T), lens.reshape(T, B).sum(1))
    idx = (rng.random(L) ** rng.choice([1, 8], L) * np.array(rows)[table]).astype(np.int32)      # runs of one to hundreds of thousands
    go = rng.standard_normal((B, T, D), dtype=np.float32)
    c = Case(wl, max_lookups=L)
    c.ctx.set_sort_path(sort_path)
    ur, uo, gr = c.gpu_bwd(idx, off, go)
    o_ur, o_uo, o_gr = oracle.emb_bwd(go, T, D, B, idx, off)
    assert bit_equal(uo, o_uo) and bit_equal(ur, o_ur)
    # n terms of magnitude below 6 in FP64 in two orders, each sum rounded once
    n = int(np.bincount(idx + 1_000_000 * table).max())
    np.testing.assert_allclose(gr, o_gr, rtol=2.0 ** -23, atol=12.0 * n * n * 2.0 ** -53)
    c.ctx.close()


# an index a bag and short bags: tiles of 8 and of 16, up to sixteen of them for a warp, and more ranges than warps
@pytest.mark.parametrize("D", [52, 60, 64])
@pytest.mark.parametrize("B,bag", [(37_700, 1), (113_700, 1), (200_003, 1), (260_000, 4)])
def test_tiles_of_large_batches(oracle, D, B, bag):
    rng = np.random.default_rng(D)
    rows = (40_000, 3, 900_000)
    T = len(rows)
    L = T * B * bag
    off = np.arange(0, L + 1, bag, dtype=np.int32)
    idx = (rng.random(L) ** rng.choice([1, 8], L) * np.repeat(rows, B * bag)).astype(np.int32)
    go = rng.standard_normal((B, T, D), dtype=np.float32)
    c = Case(W.Workload("tiles", rows, D=D, B=B, alpha=None), max_lookups=L)
    ur, uo, gr = c.gpu_bwd(idx, off, go)
    o_ur, o_uo, o_gr = oracle.emb_bwd(go, T, D, B, idx, off)
    assert bit_equal(uo, o_uo) and bit_equal(ur, o_ur)
    # as above
    n = int(np.bincount(idx + 1_000_000 * np.repeat(np.arange(T), B * bag)).max())
    np.testing.assert_allclose(gr, o_gr, rtol=2.0 ** -23, atol=12.0 * n * n * 2.0 ** -53)
    c.ctx.close()


@pytest.mark.parametrize("D,kernel", [(4, "seg_groups_kernel"), (16, "seg_groups_kernel"), (48, "seg_groups_kernel"), (52, "seg_sum_kernel"), (128, "seg_sum_kernel")])
def test_profile_names_the_kernel(D, kernel):
    """The profile says which of the two summing kernels ran."""
    B = 60
    wl = W.Workload("names", (50,), D=D, B=B, alpha=None)
    c = Case(wl)
    c.ctx.profile_begin()
    c.gpu_bwd_two_calls(np.arange(B, dtype=np.int32) % 50, np.arange(B + 1, dtype=np.int32), np.ones((B, 1, D), dtype=np.float32))
    assert set(c.ctx.profile_end()) & {"seg_groups_kernel", "seg_sum_kernel"} == {kernel}
    c.ctx.close()
