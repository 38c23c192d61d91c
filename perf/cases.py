"""Performance cases of the quantisation-aware embedding path, called as a user's program calls it.

What a program does with this package, by `mode`:

  step      one training iteration in one call (`Context.train_step`), launched eagerly
  calls     the same iteration in the four calls a loop makes whose dense layers run between forward and
            backward: `emb_fwd`, `emb_bwd`, `grad_quant_int8`, `row_update`
  pipeline  `steps` iterations over as many batches in the two-call form (`sort_batch` of the next batch beside
            `train_step_sorted` of the current one, two workspaces, two streams), replayed from one CUDA graph as
            `bench.py` does it
  host      one iteration whose batch and pooled output live in pinned host memory (`train_step_host`)
  refresh   the periodic scale refresh: min/max of every table (`scale_refresh`)
  export    bit-packed export of the tables (`pack_tables`)
  serve     an inference lookup from the packed tables (`packed_fwd`)

The shapes are those of the package's own workloads: "tiny", Kaggle-shaped (26 tables, 33.8 M rows, 16 features),
Terabyte-shaped (26 tables, 49 M rows, 64 features), multi-hot (26 tables of a million rows, about 20 indices per
bag) and the single-table sweep.  `draw` takes further shapes from the ranges these span.

Every input is made on the GPU from the seed: rows U(-1/sqrt(R), 1/sqrt(R)), indices Zipf(alpha) over the rows with the
hot rows spread over the table (alpha 0: uniform), bag lengths Poisson clipped to [1, 64], upstream gradients
N(0, 0.1^2).
"""
import math
import random

import numpy as np
import torch

import paper_2410_20046_b200 as dq

LR = 0.1
GRAD_SIGMA = 0.1
BAG_MAX = 64
MODES = ("step", "calls", "pipeline", "host", "refresh", "export", "serve")


def _case(name, mode, tables, rows, dim, batch, alpha, bag=1, bits=4, steps=1, equal=False):
    c = dict(mode=mode, tables=tables, rows=rows, dim=dim, batch=batch, alpha=alpha, bag=bag, bits=bits, steps=steps,
             equal=equal)
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # the smallest training job (four tables, a batch of 128): launches and latency are all there is
        _case("tiny_step_b128", "step", 4, 126_000, 16, 128, 1.05),
        # a Criteo Kaggle model trained with the reference recipe's small batch, dense layers between the calls
        _case("kaggle_calls_b128", "calls", 26, 33_800_000, 16, 128, 1.05),
        # the same model at a large batch, fed from a data loader's pinned buffers: bound by the host link
        _case("kaggle_host_b16384", "host", 26, 33_800_000, 16, 16_384, 1.05),
        # ... and with the batches on the device, the next batch sorted beside the current one (the benchmark's form)
        _case("kaggle_pipeline_b16384", "pipeline", 26, 33_800_000, 16, 16_384, 1.05, steps=8),
        # a Criteo Terabyte model at a middling batch, dense layers between the calls
        _case("terabyte_calls_b2048", "calls", 26, 49_000_000, 64, 2_048, 1.1),
        # ... and at the large batch, pipelined: the largest single-GPU training configuration
        _case("terabyte_pipeline_b32768", "pipeline", 26, 49_000_000, 64, 32_768, 1.1, steps=8),
        # pooled multi-hot features: about 328 thousand lookups per table, duplicate-heavy
        _case("multihot_step_b16384", "step", 26, 26_000_000, 64, 16_384, 1.2, bag=20, equal=True),
        # one very large table with wide rows, uniform indices: hardly a duplicate
        _case("sweep_step_d128_b65536", "step", 1, 10_000_000, 128, 65_536, 0.0, bits=8),
        # odd everything: feature size that fills no lane group, odd batch, short bags, 2-bit rows
        _case("ragged_calls_d36_b3001", "calls", 7, 1_234_567, 36, 3_001, 1.1, bag=3, bits=2),
        # every P-th iteration of a Kaggle-shaped job: the whole model is read once
        _case("kaggle_refresh", "refresh", 26, 33_800_000, 16, 128, 1.05),
        # end of a Kaggle-shaped job: the 4-bit model that is deployed
        _case("kaggle_export_int4", "export", 26, 33_800_000, 16, 128, 1.05),
        # the deployed Terabyte-shaped model under a large request batch
        _case("terabyte_serve_int4_b32768", "serve", 26, 49_000_000, 64, 32_768, 1.1),
    ]


def draw(rng):
    log = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))      # noqa: E731
    while True:
        mode = rng.choice(MODES)
        tables = log(1, 40)
        dim = rng.choice((8, 16, 16, 20, 32, 36, 48, 64, 64, 96, 128))
        rows = log(2e4, 4.9e7)
        batch = log(64, 65_536)
        alpha = rng.choice((0.0, 1.05, 1.1, 1.2))
        bag = rng.choice((1, 1, 1, rng.randint(2, 20)))
        bits = rng.choice((2, 4, 4, 8))
        steps = rng.choice((2, 4, 8)) if mode == "pipeline" else 1
        c = _case(None, mode, tables, rows, dim, batch, alpha, bag=bag, bits=bits, steps=steps,
                  equal=rng.random() < 0.25)
        lookups = tables * batch * bag * steps
        train = mode not in ("refresh", "export", "serve")
        if rows * dim * 4 > 12_600_000_000 or rows < 20 * tables or lookups > 6_000_000:
            continue
        if train and lookups * dim * 20 + tables * batch * dim * 8 * steps > 5_000_000_000:
            continue
        if mode in ("refresh", "export") and rows * dim * 4 > 6_000_000_000:
            continue
        if mode == "host" and tables * batch * dim * 4 > 60_000_000:
            continue
        return c


def _row_counts(case):
    """Rows per table: equal, or log-uniform in [4, 10^7] rescaled to the total (the spread of the Criteo tables)."""
    T, total = case["tables"], case["rows"]
    if case["equal"]:
        return [max(4, total // T)] * T
    r = random.Random(26)
    w = [math.exp(r.uniform(math.log(4.0), math.log(1.0e7))) for _ in range(T)]
    f = total / sum(w)
    return [max(4, int(round(f * x))) for x in w]


def _expected_unique(R, n, alpha):
    """Expected number of distinct rows among n draws from the index law over R rows."""
    if alpha == 0.0:
        return R * -math.expm1(-n / R)
    head = min(R, 4096)
    k = np.arange(1, head + 1, dtype=np.float64)
    edges = np.unique(np.concatenate([[head], np.geomspace(head, R, 2000)])) if R > head else np.array([head, head], float)
    mid, width = 0.5 * (edges[1:] + edges[:-1]), np.diff(edges)
    k, m = np.concatenate([k, mid]), np.concatenate([np.ones(head), width])
    p = k ** -alpha
    p /= (p * m).sum()
    return float((m * -np.expm1(-n * p)).sum())


def work(case):
    T, D, B = case["tables"], case["dim"], case["batch"]
    rows = _row_counts(case)
    elements = sum(rows) * D
    if case["mode"] == "refresh":
        return {"bytes": 4 * elements, "flops": 2 * elements}
    if case["mode"] == "export":
        return {"bytes": 4 * elements + elements * case["bits"] // 8, "flops": 4 * elements}
    G, n = T * B, B * case["bag"]
    L = T * n
    U = sum(_expected_unique(R, n, case["alpha"]) for R in rows)
    index = 4 * L + 4 * (G + 1)
    if case["mode"] == "serve":
        return {"bytes": index + U * D * case["bits"] / 8 + 4 * D * G, "flops": 2 * L * D}
    # pooled output written, upstream gradient read, every touched row read and written once, and the sparse
    # gradient (row numbers, FP32 sums, INT8 codes) written
    once = index + 8 * D * G + U * (8 * D + 4 + 4 * D + D)
    return {"bytes": case["steps"] * once, "flops": case["steps"] * (5 * L * D + 8 * U * D)}


def tolerance(case):
    if case["mode"] in ("refresh", "export"):
        return "exact"                 # minima, maxima, one division; integer codes
    # every sum is accumulated in FP64 and rounded once to FP32: summed in another order (measured on the tiny, the
    # Terabyte-shaped, the multi-hot and the ragged case, 90 M sums) not one result changed; a change would be a last
    # bit, 1.2e-7 of the value, in a few of 10^8 results
    return {"rel": 1e-9, "max": 2.5e-7, "differ": 1e-6}


# ---- inputs -------------------------------------------------------------------------------------------------------
def _coprime_stride(R):
    a = max(1, math.ceil(0.618 * R))
    while math.gcd(a, R) != 1:
        a += 1
    return a


def _cumulative(R, alpha):
    return torch.arange(1, R + 1, dtype=torch.float64, device="cuda").pow_(-alpha).cumsum_(0)


def _batches(case, rows, count, gen):
    """`count` batches as (indices, offsets), table-major."""
    T, B = case["tables"], case["batch"]
    lens = []
    for _ in range(count):
        if case["bag"] == 1:
            lens.append(torch.ones((T, B), dtype=torch.int64, device="cuda"))
        else:
            mean = torch.full((T, B), float(case["bag"]), device="cuda")
            lens.append(torch.poisson(mean, generator=gen).clamp_(1, BAG_MAX).to(torch.int64))
    per_table = torch.stack([x.sum(1) for x in lens]).cpu().tolist()
    parts = [[] for _ in range(count)]
    cum, cum_R = None, None
    for t, R in enumerate(rows):
        if case["alpha"] != 0.0 and R != cum_R:
            cum, cum_R = _cumulative(R, case["alpha"]), R
        for b in range(count):
            u = torch.rand(per_table[b][t], dtype=torch.float64, device="cuda", generator=gen)
            if case["alpha"] == 0.0:
                k = (u * R).to(torch.int64)
            else:
                k = torch.searchsorted(cum, u * cum[-1], right=True)
            k = k.clamp_(max=R - 1)
            parts[b].append(((k * _coprime_stride(R)) % R).to(torch.int32))
    out = []
    for b in range(count):
        off = torch.zeros(T * B + 1, dtype=torch.int32, device="cuda")
        off[1:] = lens[b].reshape(-1).cumsum(0)
        out.append((torch.cat(parts[b]), off))
    return out


def _max_lookups(case):
    bags = case["tables"] * case["batch"]
    if case["bag"] == 1:
        return bags
    mean = case["bag"] + math.exp(-case["bag"])        # empty bags are raised to one index
    return int(bags * mean + 12.0 * math.sqrt(bags * mean)) + 64


def _tables(case, rows, gen):
    arena = torch.empty((sum(rows), case["dim"]), dtype=torch.float32, device="cuda")
    at = 0
    for R in rows:
        a = 1.0 / math.sqrt(R)
        arena[at:at + R].uniform_(-a, a, generator=gen)
        at += R
    return arena


class _State:
    pass


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    T, D, B, mode = case["tables"], case["dim"], case["batch"], case["mode"]
    s = _State()
    s.mode, s.B = mode, B
    rows = _row_counts(case)
    off = [0]
    for r in rows:
        off.append(off[-1] + r)
    s.tables = _tables(case, rows, gen)
    s.bits = torch.full((T,), case["bits"], dtype=torch.int32, device="cuda")
    s.scales = torch.zeros(T, dtype=torch.float32, device="cuda")
    if mode in ("refresh", "export"):
        s.ctx = dq.Context(off, D, 1, T)
        s.minmax = torch.zeros((T, 2), dtype=torch.float32, device="cuda")
        if mode == "export":
            s.pack_bits = case["bits"]
            s.ctx.scale_refresh(s.tables, s.bits, s.scales)
            s.packed = torch.zeros(s.ctx.packed_bytes(case["bits"]), dtype=torch.uint8, device="cuda")
        return s
    s.batches = _batches(case, rows, case["steps"], gen)
    s.L = [int(i.numel()) for i, _ in s.batches]
    L = _max_lookups(case)                 # a program sizes its buffers for the largest batch it may get
    s.ctx = dq.Context(off, D, L, T * B, host_step=(mode == "host"))
    s.ctx.scale_refresh(s.tables, s.bits, s.scales)
    s.out = torch.zeros((B, T, D), dtype=torch.float32, device="cuda")
    if mode == "serve":
        s.pack_bits = case["bits"]
        s.packed = torch.empty(s.ctx.packed_bytes(case["bits"]), dtype=torch.uint8, device="cuda")
        s.ctx.pack_tables(s.tables, s.scales, case["bits"], s.packed)
        s.tables = None                # a serving process holds the packed model only
        return s
    s.grads = [torch.randn((B, T, D), dtype=torch.float32, device="cuda", generator=gen).mul_(GRAD_SIGMA)
               for _ in s.batches]
    if mode == "host":
        s.h_idx, s.h_off = (x.cpu().pin_memory() for x in s.batches[0])
        s.h_grad = s.grads[0].cpu().pin_memory()
        s.h_out = torch.zeros((B, T, D), dtype=torch.float32).pin_memory()
        s.batches = s.grads = s.out = None
        return s
    s.ur = [torch.zeros(L, dtype=torch.int32, device="cuda") for _ in range(2)]
    s.uo = [torch.zeros(T + 1, dtype=torch.int32, device="cuda") for _ in range(2)]
    s.gr = torch.zeros((L, D), dtype=torch.float32, device="cuda")
    s.codes = torch.zeros((L, D), dtype=torch.int8, device="cuda")
    s.gs = torch.zeros(T, dtype=torch.float32, device="cuda")
    if mode == "pipeline":
        _capture(s)
    return s


def _capture(s):
    """The steps of the pipelined loop, captured once into a CUDA graph."""
    train, side = torch.cuda.Stream(priority=-1), torch.cuda.Stream(priority=0)
    n = len(s.batches)

    def sort(k):
        idx, off = s.batches[k]
        s.ctx.sort_batch(idx, off, s.ur[k & 1], s.uo[k & 1], B=s.B, L=s.L[k], ws=k & 1, stream=side)

    def step(k, lr):
        idx, off = s.batches[k]
        s.ctx.train_step_sorted(s.tables, idx, off, s.grads[k], s.scales, s.bits, s.out, s.ur[k & 1], s.uo[k & 1],
                                s.gr, s.codes, s.gs, lr, B=s.B, L=s.L[k], ws=k & 1, stream=train)

    def loop(lr):
        side.wait_stream(train)
        sort(0)
        for k in range(n):
            if k + 1 < n:
                side.wait_stream(train)        # the workspace it sorts into was read by the step before
                sort(k + 1)
            step(k, lr)
        train.wait_stream(side)

    train.wait_stream(torch.cuda.current_stream())
    loop(0.0)                                  # first use outside the capture; a zero rate leaves the tables as they are
    torch.cuda.synchronize()
    s.graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(s.graph, stream=train):
        loop(LR)
    for x in s.ur + s.uo + [s.out, s.gr, s.codes, s.gs]:
        x.zero_()


# ---- one pass -------------------------------------------------------------------------------------------------------
def run(s):
    ctx, B = s.ctx, s.B
    if s.mode == "refresh":
        ctx.scale_refresh(s.tables, s.bits, s.scales, s.minmax)
        return s.scales, s.minmax
    if s.mode == "export":
        ctx.pack_tables(s.tables, s.scales, s.pack_bits, s.packed)
        return s.packed
    if s.mode == "host":
        ctx.train_step_host(s.tables, s.h_idx, s.h_off, s.h_grad, s.scales, s.bits, s.h_out, LR, B=B, L=s.L[0])
        return s.h_out, s.tables
    if s.mode == "pipeline":
        s.graph.replay()
        return s.out, s.ur, s.uo, s.gr, s.codes, s.gs, s.tables
    idx, off = s.batches[0]
    L = s.L[0]
    if s.mode == "serve":
        ctx.packed_fwd(s.packed, idx, off, s.scales, s.pack_bits, s.out, B=B, L=L)
        return s.out
    ur, uo, grad = s.ur[0], s.uo[0], s.grads[0]
    if s.mode == "step":
        ctx.train_step(s.tables, idx, off, grad, s.scales, s.bits, s.out, ur, uo, s.gr, s.codes, s.gs, LR, B=B, L=L)
    else:
        ctx.emb_fwd(s.tables, idx, off, s.scales, s.bits, s.out, B=B, L=L)
        ctx.emb_bwd(grad, idx, off, ur, uo, s.gr, B=B, L=L)
        ctx.grad_quant_int8(s.gr, uo, s.codes, s.gs)
        ctx.row_update(s.tables, ur, uo, s.codes, s.gs, LR)
    return s.out, ur, uo, s.gr, s.codes, s.gs, s.tables
