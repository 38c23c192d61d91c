"""The one-call step and the two-call loop captured into a CUDA graph give, replayed, the bits of the same calls made one by one:
on the caller's stream alone, forked, and with each half on a stream of the context."""
import pytest

from dqrm_inputs import workloads as W
from gpu_util import Case, bit_equal

pytestmark = pytest.mark.gpu


# tables, bags, indices a bag, features: one launch behind the forward, a chain, forked (an index a bag and not), backward aside,
# forward on the caller's stream, a radix sort, a table alone by its parts
@pytest.mark.parametrize("T,B,bag,D", [(4, 100, 1, 16), (4, 700, 1, 16), (3, 900, 3, 16), (6, 1_100, 1, 64), (26, 2_000, 1, 16), (3, 50_000, 1, 128), (1, 70_000, 64, 64),
                                         (1, 50_001, 1, 16), (1, 60_000, 1, 64)])
@pytest.mark.parametrize("two_calls", [False, True])
def test_captured_steps(T, B, bag, D, two_calls):
    import torch

    wl = W.Workload("captured", (5_000,) * T, D=D, B=B, alpha=None)
    L, rows, steps = T * B * bag, min(T * B * bag, 5_000 * T), 3
    c = Case(wl, max_lookups=L)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(B)
    tables = torch.rand((wl.total_rows, D), device="cuda", generator=gen) - 0.5
    batches = [(torch.randint(0, 5_000, (L,), device="cuda", generator=gen, dtype=torch.int32),
                torch.randn((B, T, D), device="cuda", generator=gen)) for _ in range(steps)]
    off = torch.arange(0, L + 1, bag, dtype=torch.int32, device="cuda")
    scales = torch.zeros(T, device="cuda")
    c.ctx.scale_refresh(tables, c.bits, scales)
    w, out = tables.clone(), [torch.zeros((B, T, D), device="cuda") for _ in range(steps)]
    ur = [torch.zeros(L, dtype=torch.int32, device="cuda") for _ in range(2)]
    uo = [torch.zeros(T + 1, dtype=torch.int32, device="cuda") for _ in range(2)]
    gr, codes, gs = torch.zeros((rows, D), device="cuda"), torch.zeros((rows, D), dtype=torch.int8, device="cuda"), torch.zeros(T, device="cuda")
    side = torch.cuda.Stream()

    def loop():
        cur = torch.cuda.current_stream()
        for k, (idx, go) in enumerate(batches):
            if not two_calls:
                c.ctx.train_step(w, idx, off, go, scales, c.bits, out[k], ur[0], uo[0], gr, codes, gs, 0.1, B=B, L=L)
                continue
            for j in ([0] if k == 0 else []) + ([k + 1] if k + 1 < steps else []):       # the next batch beside the current one
                side.wait_stream(cur)
                c.ctx.sort_batch(batches[j][0], off, ur[j & 1], uo[j & 1], B=B, L=L, ws=j & 1, stream=side)
            c.ctx.train_step_sorted(w, idx, off, go, scales, c.bits, out[k], ur[k & 1], uo[k & 1], gr, codes, gs, 0.1, B=B, L=L, ws=k & 1)
        if two_calls:
            cur.wait_stream(side)

    seen = []

    def look():
        torch.cuda.synchronize()
        c.ctx.raise_on_device_error()
        last = (steps - 1) & 1 if two_calls else 0
        U = int(uo[last][-1])
        seen.append([x.cpu().numpy() for x in (w, *out, ur[last][:U], uo[last], gr[:U], codes[:U], gs)])

    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        loop()
    look()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        loop()
    for _ in range(2):
        w.copy_(tables)
        for x in out + ur + uo + [gr, codes, gs]:
            x.zero_()
        torch.cuda.synchronize()
        graph.replay()
        look()
    for replayed in seen[1:]:
        for a, b in zip(seen[0], replayed):
            assert bit_equal(a, b)
    del graph
    c.ctx.close()
