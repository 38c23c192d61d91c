"""GPU parity of the one-launch gradient quantiser at its edges: tables of no, one and many rows, sizes around what the
blocks of a cluster hold in registers, a table far larger than that beside small ones, and buffers so large that the
quantiser of three launches takes over."""
import numpy as np
import pytest

from dqrm_inputs import workloads as W
from gpu_util import Case, bit_equal

pytestmark = pytest.mark.gpu

# rows per table, and the rows the buffers have room for (None: just these)
SHAPES = {
    (4, "tiny"): ([0, 1, 511, 512, 513, 0], None),
    (16, "around one block"): ([128, 127, 129, 0, 1024, 1025], None),
    (64, "one table"): ([2048], None),
    (64, "what a cluster holds"): ([2047, 2048, 2049], None),
    (64, "one table holds nearly all"): ([0, 9000, 1, 0, 0, 0, 3, 0], None),
    (1020, "wide rows"): ([5, 0, 70], None),
    (16, "larger than the registers"): ([9000] * 10 + [0, 200] * 5, None),
    (64, "blocks of 1024"): ([4096, 2050, 0, 1], None),
    (16, "large buffers"): ([128, 0, 700], 300_000),
    # tables beyond what their cluster takes, which all blocks share
    (64, "one of many shared"): ([0, 30_000, 1, 0, 3] + [40] * 21, None), (36, "two shared"): ([20_000, 7, 0, 20_000] + [9] * 22, None),
    (16, "few tables, one shared"): ([40_000, 1, 0], None), (64, "just not shared"): ([0, 2048, 0, 0, 0, 0, 0, 0], None),
    (64, "just shared"): ([0, 2049, 0, 0, 0, 0, 0, 0], None), (20, "last one shared"): ([1] * 150 + [9_000], None),
}


@pytest.mark.parametrize("shape", list(SHAPES))
def test_quant_table(oracle, shape):
    D, (rows, room) = shape[0], SHAPES[shape]
    wl = W.Workload("quant", (10_000,) * len(rows), D=D, B=4, alpha=None)
    rng = np.random.default_rng(sum(rows) + D)
    uo = np.concatenate([[0], np.cumsum(rows)]).astype(np.int32)
    gr = rng.standard_normal((int(uo[-1]), D)).astype(np.float32) * 10.0 ** rng.integers(-6, 6, (int(uo[-1]), 1))
    gr = gr.astype(np.float32)
    gr[::17] = 0.0
    o_codes, o_gs = oracle.grad_quant_int8(gr, uo, D)
    c = Case(wl, max_lookups=int(uo[-1]))
    t = c.torch
    n = room or len(gr)
    d_gr, d_codes = t.full((n, D), 1e30, device="cuda"), t.full((n, D), 99, dtype=t.int8, device="cuda")
    d_gr[:len(gr)] = c.dev(gr)
    gs = c.empty(wl.T, t.float32)
    c.ctx.grad_quant_int8(d_gr, c.dev(uo), d_codes, gs)
    codes = d_codes.cpu().numpy()
    assert bit_equal(gs.cpu().numpy(), o_gs) and bit_equal(codes[:len(gr)], o_codes)
    assert (codes[len(gr):] == 99).all()
    c.ctx.close()


@pytest.mark.parametrize("rows,most", [([0, 30_000, 1, 0, 3] + [40] * 21, None), ([0, 30_000, 1, 0, 3] + [40] * 21, 64),
                                       ([128, 3], 0), ([128, 3], 1 << 40)])
def test_neither_the_bound_nor_the_workspace_changes_the_result(oracle, rows, most):
    """A bound that is too small or too large, and a workspace of the least size that was ever asked for."""
    D = 64
    wl = W.Workload("quant", (100_000,) * len(rows), D=D, B=4, alpha=None)
    rng = np.random.default_rng(len(rows))
    uo = np.concatenate([[0], np.cumsum(rows)]).astype(np.int32)
    gr = rng.standard_normal((int(uo[-1]), D)).astype(np.float32)
    o_codes, o_gs = oracle.grad_quant_int8(gr, uo, D)
    c = Case(wl, max_lookups=len(gr))
    t = c.torch
    d_gr, d_uo, codes, gs = c.dev(gr), c.dev(uo), c.empty((len(gr), D), t.int8), c.empty(wl.T, t.float32)
    for room in (256, c.ctx.scratch_bytes):
        codes.fill_(99)
        assert c.ctx.lib.dqrm_grad_quant_int8_bounded(
            c.ctx._h, d_gr.data_ptr(), d_uo.data_ptr(), codes.data_ptr(), gs.data_ptr(), gr.size if most is None else most,
            c.ctx._scratch_ptr, room, t.cuda.current_stream().cuda_stream) == 0
        assert bit_equal(gs.cpu().numpy(), o_gs) and bit_equal(codes.cpu().numpy(), o_codes)
    c.ctx.close()
