"""The summed gradient of rows that begin on 4 or 8 bytes, as far as the call takes them, is bit for bit that of aligned rows, and
nothing beside them is written."""
import numpy as np
import pytest

from dqrm_inputs import workloads as W
from gpu_util import Case, bit_equal

pytestmark = pytest.mark.gpu


def placed(torch, shape, dtype, offset, fill):
    """A tensor whose data begins `offset` elements behind an aligned address, with guards of `fill` around it."""
    n = int(np.prod(shape))
    buf = torch.full((n + 64,), fill, dtype=dtype, device="cuda")
    assert buf.data_ptr() % 256 == 0
    return buf, buf[32 + offset:32 + offset + n].view(shape)


@pytest.mark.parametrize("D,offset", [(4, 1), (4, 2), (4, 3), (8, 2), (12, 2), (16, 2), (20, 2), (32, 2), (36, 2), (48, 2), (52, 2), (64, 2)])
@pytest.mark.parametrize("B", [5, 700])
def test_sum_of_rows_that_are_not_aligned(oracle, B, D, offset):
    import torch

    T = 3
    wl = W.Workload("aligned", (50, 4_000, 7), D=D, B=B, alpha=None)
    rng = np.random.default_rng(B + D)
    lens = rng.integers(0, 6, T * B)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    table = np.repeat(np.arange(T), lens.reshape(T, B).sum(1))
    idx = (rng.random(off[-1]) * np.array(wl.rows)[table]).astype(np.int32)
    L = len(idx)
    go = rng.standard_normal((B, T, D)).astype(np.float32)
    c = Case(wl, max_lookups=L)
    ur, uo, gr = c.gpu_bwd(idx, off, go)
    o_ur, o_uo, o_gr = oracle.emb_bwd(go, T, D, B, idx, off)
    assert bit_equal(uo, o_uo) and bit_equal(ur, o_ur)
    # at most L terms of magnitude below 6 in FP64 in two orders, each sum rounded once
    np.testing.assert_allclose(gr, o_gr, rtol=2.0 ** -23, atol=12.0 * L ** 2 * 2.0 ** -53)
    U = len(ur)
    d_idx, d_off = c.dev(idx), c.dev(off)
    for go_off, gr_off in ((offset, 0), (0, offset), (offset, offset)):
        go_buf, d_go = placed(torch, (B, T, D), torch.float32, go_off, 1e30)
        d_go.copy_(torch.from_numpy(go))
        gr_buf, d_gr = placed(torch, (L, D), torch.float32, gr_off, -7.0)
        d_ur, d_uo = c.empty(L, torch.int32), c.empty(T + 1, torch.int32)
        c.ctx.emb_bwd(d_go, d_idx, d_off, d_ur, d_uo, d_gr, B=B, L=L)
        c.ctx.raise_on_device_error()
        assert bit_equal(d_gr[:U].cpu().numpy(), gr) and bit_equal(d_ur[:U].cpu().numpy(), ur) and bit_equal(d_uo.cpu().numpy(), uo)
        rest = gr_buf.cpu().numpy()
        rest[32 + gr_off:32 + gr_off + U * D] = -7.0
        assert (rest == -7.0).all()
    # the step, whose upstream gradient alone may lie so
    tables = torch.rand((wl.total_rows, D), device="cuda") - 0.5
    scales = c.empty(T, torch.float32)
    c.ctx.scale_refresh(tables, c.bits, scales)
    seen = []
    for by in (0, offset):
        w = tables.clone()
        d_go = placed(torch, (B, T, D), torch.float32, by, 1e30)[1]
        d_go.copy_(torch.from_numpy(go))
        out, d_gr, codes = c.empty((B, T, D), torch.float32), c.empty((L, D), torch.float32), c.empty((L, D), torch.int8)
        gs = c.empty(T, torch.float32)
        c.ctx.train_step(w, d_idx, d_off, d_go, scales, c.bits, out, d_ur, d_uo, d_gr, codes, gs, 0.1, B=B, L=L)
        c.ctx.raise_on_device_error()
        seen.append([x.cpu().numpy() for x in (w, out, d_ur[:U], d_uo, codes[:U], gs)])
    for a, b in zip(*seen):
        assert bit_equal(a, b)
    c.ctx.close()
