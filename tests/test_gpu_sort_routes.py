"""Which blocks sort a batch in the two-call and the host-fed step, where the sort runs beside a training step: a table alone by its
parts, whose four lists go from dqrm_sort_batch to dqrm_train_step_sorted, and many tables on both sides of the lines; and unusable
boundaries in each of these sorts."""
import numpy as np
import pytest

from dqrm_inputs import workloads as W
from gpu_util import Case, assert_close_fp32, bit_equal

pytestmark = pytest.mark.gpu


def batches(wl, L, n, seed):
    """n batches with gradients whose sums are exact (multiples of 2^-8 below 4, sums of less than 2^16 of them), so every output has one value"""
    rng = np.random.default_rng(seed)
    off = np.arange(L + 1, dtype=np.int32)
    out = []
    for k in range(n):
        idx = np.concatenate([rng.integers(0, R, wl.B) if k % 2 else (R ** rng.random(wl.B)).astype(np.int64).clip(0, R - 1) for R in wl.rows])
        out.append((idx.astype(np.int32), off, (rng.integers(-1024, 1025, (wl.B, wl.T, wl.D)) / 256).astype(np.float32)))
    return out


# rows of which quarters take a pass less, of three passes, of two; the fewest lookups that are shared, and large batches
@pytest.mark.parametrize("D", [16, 64])
@pytest.mark.parametrize("rows,L", [(200_000, 16_384), (3_000_000, 16_384), (3_000_000, 65_536), (60_000, 49_152), (3, 50_000)])
def test_table_alone_in_two_calls(oracle, rows, L, D):
    import torch

    wl = W.Workload("alone", (rows,), D=D, B=L, alpha=None)
    c = Case(wl)
    o_tables = W.tables_np(wl)
    d_tables, scales = c.dev(o_tables), c.empty(1, torch.float32)
    c.ctx.scale_refresh(d_tables, c.bits, scales)
    o_scales, _ = oracle.scale_refresh(o_tables, c.row_off, D, c.bits_np)
    steps = batches(wl, L, 3, rows + D)
    dev = [tuple(c.dev(a) for a in b) for b in steps]
    ur, uo = [c.empty(L, torch.int32) for _ in range(2)], [c.empty(2, torch.int32) for _ in range(2)]
    out, gr, codes, gs = c.empty((L, 1, D), torch.float32), c.empty((L, D), torch.float32), c.empty((L, D), torch.int8), c.empty(1, torch.float32)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    c.ctx.sort_batch(*dev[0][:2], ur[0], uo[0], B=L, L=L, ws=0, stream=side)
    for k, (idx, off, go) in enumerate(dev):
        torch.cuda.current_stream().wait_stream(side)
        if k + 1 < len(dev):
            side.wait_stream(torch.cuda.current_stream())
            c.ctx.sort_batch(*dev[k + 1][:2], ur[(k + 1) & 1], uo[(k + 1) & 1], B=L, L=L, ws=(k + 1) & 1, stream=side)
        c.ctx.train_step_sorted(d_tables, idx, off, go, scales, c.bits, out, ur[k & 1], uo[k & 1], gr, codes, gs, wl.lr, B=L, L=L, ws=k & 1)
        r = oracle.train_step(o_tables, c.row_off, D, L, *steps[k], o_scales, c.bits_np, wl.lr)
        U = int(r["uniq_off"][-1])
        assert bit_equal(uo[k & 1].cpu().numpy(), r["uniq_off"]) and bit_equal(ur[k & 1].cpu().numpy()[:U], r["unique_rows"])
        assert bit_equal(gr.cpu().numpy()[:U], r["grad_rows"])
        assert bit_equal(gs.cpu().numpy(), r["grad_scales"]) and bit_equal(codes.cpu().numpy()[:U], r["codes"])
        assert_close_fp32(out.cpu().numpy(), r["out"])
    c.ctx.raise_on_device_error()
    assert bit_equal(d_tables.cpu().numpy(), o_tables)
    c.ctx.close()


@pytest.mark.parametrize("rows,L,D", [(200_000, 17_001, 16), (3_000_000, 40_000, 64), (60_000, 50_000, 20)])
def test_table_alone_fed_by_the_host(oracle, rows, L, D):
    import torch

    wl = W.Workload("alone", (rows,), D=D, B=L, alpha=None)
    c = Case(wl, host_step=True)
    o_tables = W.tables_np(wl)
    d_tables, scales = c.dev(o_tables), c.empty(1, torch.float32)
    c.ctx.scale_refresh(d_tables, c.bits, scales)
    o_scales, _ = oracle.scale_refresh(o_tables, c.row_off, D, c.bits_np)
    steps = batches(wl, L, 3, rows + D)
    pinned = [tuple(torch.from_numpy(a).pin_memory() for a in b) for b in steps]
    outs = [torch.empty((L, 1, D)).pin_memory() for _ in steps]
    torch.cuda.synchronize()
    for (idx, off, go), out in zip(pinned, outs):
        c.ctx.train_step_host(d_tables, idx, off, go, scales, c.bits, out, wl.lr, B=L, L=L)
    torch.cuda.synchronize()
    c.ctx.raise_on_device_error()
    for b, out in zip(steps, outs):
        r = oracle.train_step(o_tables, c.row_off, D, L, *b, o_scales, c.bits_np, wl.lr)
        assert_close_fp32(out.numpy(), r["out"])
    assert bit_equal(d_tables.cpu().numpy(), o_tables)
    c.ctx.close()


# clusters of eight, of four, and of eight of which half works: tables, features, lookups a table on both sides of the lines beside a step
@pytest.mark.parametrize("even", [True, False])
@pytest.mark.parametrize("T,D,per_table", [(18, 36, 2_600), (19, 36, 2_600), (19, 36, 8_192), (19, 36, 8_193), (19, 16, 2_560), (19, 16, 2_561),
                                           (34, 16, 2_600), (37, 16, 8_192), (38, 8, 8_193)])
def test_many_tables_beside_a_step(oracle, T, D, per_table, even):
    rng = np.random.default_rng(T + per_table)
    rows = tuple(int(r) for r in rng.choice([1, 300, 70_000], T))
    B = per_table
    lens = np.ones((T, B), dtype=np.int64)
    if not even:
        lens[0] = 3                      # one table of three times the mean
        lens[1, 1:] = 0
        lens[2, 1:] = 0
        lens[2, 0] = 0                   # (fewer lookups than bags)
    off = np.concatenate([[0], np.cumsum(lens.reshape(-1))]).astype(np.int32)
    idx = np.concatenate([rng.integers(0, rows[t], n) for t, n in enumerate(lens.sum(1))]).astype(np.int32)
    go = rng.standard_normal((B, T, D), dtype=np.float32)
    c = Case(W.Workload("beside", rows, D=D, B=B, alpha=None), max_lookups=len(idx))
    ur, uo, gr = c.gpu_bwd_two_calls(idx, off, go, ws=1)
    o_ur, o_uo, o_gr = oracle.emb_bwd(go, T, D, B, idx, off)
    assert bit_equal(uo, o_uo) and bit_equal(ur, o_ur)
    # n terms of magnitude below 6 in FP64 in two orders, each sum rounded once
    n = int(np.bincount(idx + 100_000 * np.repeat(np.arange(T), lens.sum(1))).max())
    np.testing.assert_allclose(gr, o_gr, rtol=2.0 ** -23, atol=12.0 * n * n * 2.0 ** -53)
    c.ctx.close()


# small batches, a table alone by its parts (first and last offset), clusters of four, clusters of eight of which half works (a boundary inside, too)
@pytest.mark.parametrize("T,B,bag,where", [(3, 100, 1, "inside"), (1, 20_000, 1, "first"), (1, 20_000, 1, "last"), (20, 2_500, 1, "first"), (20, 2_500, 1, "inside"),
                                           (20, 2_500, 1, "last"), (40, 1_500, 2, "first"), (40, 1_500, 2, "inside"), (40, 1_500, 2, "last")])
@pytest.mark.parametrize("calls", ["bwd", "two"])
def test_unusable_boundaries(oracle, T, B, bag, where, calls):
    """Reported; nothing is summed, no row changes, no scale but that of an empty gradient; and the context stays usable."""
    import torch
    import paper_2410_20046_b200 as dq

    D, L = 16, T * B * bag
    wl = W.Workload("boundaries", (300_000,) + (50,) * (T - 1), D=D, B=B, alpha=None)
    c = Case(wl, max_lookups=L)
    rng = np.random.default_rng(T)
    off = np.arange(0, L + 1, bag, dtype=np.int32)
    bad = off.copy()
    at, value = {"first": (0, 5), "inside": ((7 if T > 7 else 1) * B, L + 3), "last": (T * B, L - 1)}[where]
    bad[at] = value
    idx = rng.integers(0, 50, L).astype(np.int32)
    go = rng.standard_normal((B, T, D)).astype(np.float32)
    ur, uo = torch.full((L,), -1, dtype=torch.int32, device="cuda"), torch.full((T + 1,), -1, dtype=torch.int32, device="cuda")
    gr = torch.full((L, D), 7.0, device="cuda")
    if calls == "bwd":
        c.ctx.emb_bwd(c.dev(go), c.dev(idx), c.dev(bad), ur, uo, gr, B=B, L=L)
    else:
        tables = W.tables_np(wl)
        d_tables, scales, out = c.dev(tables), c.dev(np.full(T, 0.1, np.float32)), c.empty((B, T, D), torch.float32)
        codes, gs = c.empty((L, D), torch.int8), c.empty(T, torch.float32)
        c.ctx.sort_batch(c.dev(idx), c.dev(bad), ur, uo, B=B, L=L)
        c.ctx.train_step_sorted(d_tables, c.dev(idx), c.dev(bad), c.dev(go), scales, c.bits, out, ur, uo, gr, codes, gs, 0.1, B=B, L=L)
    with pytest.raises(dq.DqrmError) as e:
        c.ctx.raise_on_device_error()
    assert e.value.status == dq.ERR_INDEX_RANGE
    assert not uo.cpu().numpy().any()
    assert (gr.cpu().numpy() == 7.0).all() and (ur.cpu().numpy() == -1).all()
    if calls == "two":
        assert (gs.cpu().numpy() == oracle.scale_from_absmax(0.0, 8)).all() and bit_equal(d_tables.cpu().numpy(), tables)
    assert c.ctx.check_status() == dq.OK
    g_ur, g_uo, g_gr = c.gpu_bwd(idx, off, go)
    o_ur, o_uo, o_gr = oracle.emb_bwd(go, T, D, B, idx, off)
    assert bit_equal(g_ur, o_ur) and bit_equal(g_uo, o_uo)
    assert_close_fp32(g_gr, o_gr)
    c.ctx.close()
