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
