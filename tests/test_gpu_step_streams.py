"""The one-call step gives the same bits whichever of its halves runs on a stream of the context: batches on both sides of
the sizes (bytes of gathered rows) at which the halves change streams, several steps in a row without a wait between."""
import numpy as np
import pytest

from dqrm_inputs import workloads as W
from gpu_util import Case, bit_equal

pytestmark = pytest.mark.gpu

MB = 1 << 20


# tables, bags, indices a bag, features
@pytest.mark.parametrize("T,B,bag,D", [
    (2, 2_047, 1, 64), (2, 2_048, 1, 64),              # 1 MB
    (3, 43_690, 1, 128), (3, 43_691, 1, 128),          # 64 MB
    (1, 65_535, 64, 64), (1, 65_536, 64, 64),          # 1 GB
])
def test_streams_do_not_matter(T, B, bag, D):
    import torch

    wl = W.Workload("streams", (5_000,) * T, D=D, B=B, alpha=None)
    L = T * B * bag
    c = Case(wl, max_lookups=L)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(B)
    tables = torch.rand((wl.total_rows, D), device="cuda", generator=gen) - 0.5
    batches = []
    for _ in range(2):
        idx = torch.randint(0, 5_000, (L,), device="cuda", generator=gen, dtype=torch.int32)
        batches.append((idx, torch.randn((B, T, D), device="cuda", generator=gen)))
    off = torch.arange(0, L + 1, bag, dtype=torch.int32, device="cuda")
    scales = torch.zeros(T, device="cuda")
    c.ctx.scale_refresh(tables, c.bits, scales)
    seen = []
    for overlap in (True, False):
        c.ctx.set_overlap(overlap)
        w = tables.clone()
        outs = [torch.empty((B, T, D), device="cuda") for _ in range(3)]
        ur, uo, gr = (torch.zeros(L, dtype=torch.int32, device="cuda"), torch.zeros(T + 1, dtype=torch.int32, device="cuda"),
                      torch.zeros((T * 5_000, D), device="cuda"))
        codes, gs = torch.zeros((T * 5_000, D), dtype=torch.int8, device="cuda"), torch.zeros(T, device="cuda")
        for k in range(3):
            c.ctx.train_step(w, batches[k & 1][0], off, batches[k & 1][1], scales, c.bits, outs[k], ur, uo, gr, codes, gs,
                             0.1, B=B, L=L)
        c.ctx.raise_on_device_error()
        U = int(uo[-1])
        seen.append([x.cpu().numpy() for x in (w, *outs, ur[:U], uo, gr[:U], codes[:U], gs)])
    for a, b in zip(*seen):
        assert bit_equal(a, b)
    c.ctx.close()


@pytest.mark.parametrize("T,B,D", [
    (2, 8_191, 16), (2, 8_192, 16), (2, 3_640, 36), (2, 3_641, 36),                  # 1 MB
    (4, 262_143, 16), (4, 262_144, 16), (2, 233_016, 36), (2, 233_017, 36),          # 64 MB
])
def test_streams_do_not_matter_to_lane_groups(T, B, D):
    test_streams_do_not_matter(T, B, 1, D)
