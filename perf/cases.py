"""The work that users of this package have it do, as cases that can be timed and compared.

Every case goes through the public binding (``paper_2412_04180_b200.skim.Skim``) the way a program
does: a context with a workspace for the matrix's size, the matrix and its importances on the GPU (in pinned host memory
for the host-buffer entry point), output buffers kept where a program keeps them.  The matrices follow the
recipe of ``paper_2412_04180_b200/inputs.py`` (N(0, 0.02) weights in binary16 with 0.1 % of
heavy-tailed outliers, log-normal importances), drawn on the GPU.  Sizes are the LLaMA layer shapes of the benchmark's
configurations, its 256 x 512 first configuration, and ragged ones.

Kinds of work:

* ``pipeline``   cluster every row at every width, allocate bits, emit packed codes and codebooks
* ``alternate``  one round of the grouping/scaling alternation: install alpha, re-cluster at the allocated
                 widths with labels, Adam steps on alpha (diagonal loss)
* ``lfull_alternate``  the same round with the paper's L-full loss
* ``lfull_table``  the L-full error table of all widths and the allocation from it
* ``exact``      optimal clustering of every row at every width
* ``host``       the whole path from pinned host buffers to pinned host buffers
* ``dequantize``, ``matvec``  the consumers of the packed form
"""
from __future__ import annotations

import math

import torch

from paper_2412_04180_b200.skim import Skim

ITERS = 50


def listed():
    return [
        # the first configuration: the smallest matrix anyone tries, bound by launches and latency
        dict(name="pipeline 256x512", kind="pipeline", rows=256, cols=512, bit_min=1, iters=30, budget=3.2, scaled=False),
        # a row length no vector load divides (unaligned rows), few rows
        dict(name="pipeline 1000x3001", kind="pipeline", rows=1000, cols=3001, bit_min=1, iters=ITERS, budget=2.25, scaled=False),
        # LLaMA-7B attention projection: four of a block's seven matrices
        dict(name="pipeline 4096x4096", kind="pipeline", rows=4096, cols=4096, bit_min=1, iters=ITERS, budget=3.0, scaled=False),
        # LLaMA-7B down projection: the benchmark's matrix
        dict(name="pipeline 4096x11008", kind="pipeline", rows=4096, cols=11008, bit_min=1, iters=ITERS, budget=3.0, scaled=False),
        # one alternation round of the same matrix, the paper's 120 Adam steps
        dict(name="alternate 4096x11008", kind="alternate", rows=4096, cols=11008, bit_min=1, iters=ITERS, budget=3.0, steps=120),
        # LLaMA-65B gate/up projection: the largest matrix of the configurations
        dict(name="alternate 22016x8192", kind="alternate", rows=22016, cols=8192, bit_min=1, iters=ITERS, budget=3.0, steps=120),
        # the round with the loss the paper uses in it
        dict(name="lfull_alternate 4096x4096", kind="lfull_alternate", rows=4096, cols=4096, bit_min=1, iters=ITERS, budget=3.0,
             steps=120),
        # the error table in the paper's form
        dict(name="lfull_table 4096x11008", kind="lfull_table", rows=4096, cols=11008, bit_min=1, budget=3.0),
        # optimal clustering of a sample of rows, to judge the iterations by
        dict(name="exact 256x4096", kind="exact", rows=256, cols=4096, bit_min=1),
        # a program whose checkpoint lies in host memory
        dict(name="host 4096x11008", kind="host", rows=4096, cols=11008, bit_min=1, iters=ITERS, budget=3.0),
        # fp16 weights back from the packed form (prefill through a dense GEMM), alpha applied
        dict(name="dequantize 4096x11008", kind="dequantize", rows=4096, cols=11008, bit_min=1, budget=3.0, scaled=True),
        # one decoded token
        dict(name="matvec 4096x11008", kind="matvec", rows=4096, cols=11008, bit_min=1, budget=3.0, scaled=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, rows, cols, elements, step=1):
    """Log-uniform rows and cols (cols a multiple of ``step``), at most ``elements`` of them together."""
    c = max(cols[0], min(cols[1], _log_int(rng, *cols) // step * step))
    r = _log_int(rng, rows[0], max(rows[0], min(rows[1], elements // c)))
    return r, c


# what is run most is drawn most
_KINDS = ["pipeline"] * 4 + ["alternate"] * 2 + ["lfull_alternate", "lfull_table", "exact", "host"] + ["dequantize"] * 2 + ["matvec"] * 2


def draw(rng):
    kind = rng.choice(_KINDS)
    bit_min = rng.choice([1, 1, 1, 2])
    budget = round(rng.uniform(bit_min + 1, 3.5), 2)
    scaled = rng.random() < 0.5
    # model rows are multiples of 8 elements far more often than not
    step = rng.choice([1, 8])
    if kind in ("pipeline", "host"):
        rows, cols = _size(rng, (64, 22016), (128, 22016), 22016 * 8192 if kind == "pipeline" else 4096 * 11008, step)
        case = dict(kind=kind, rows=rows, cols=cols, bit_min=bit_min, iters=rng.choice([20, 30, 50, 50]), budget=budget)
        return dict(case, scaled=scaled) if kind == "pipeline" else case
    if kind == "alternate":
        rows, cols = _size(rng, (512, 22016), (128, 22016), 22016 * 8192, step)
        return dict(kind=kind, rows=rows, cols=cols, bit_min=bit_min, iters=ITERS, budget=budget, steps=rng.choice([20, 40, 120]))
    if kind == "lfull_alternate":
        rows, cols = _size(rng, (512, 8192), (256, 11008), 4096 * 8192, 8)
        return dict(kind=kind, rows=rows, cols=cols, bit_min=bit_min, iters=ITERS, budget=budget, steps=rng.choice([20, 40]))
    if kind == "lfull_table":
        rows, cols = _size(rng, (128, 11008), (256, 11008), 4096 * 11008, 8)
        return dict(kind=kind, rows=rows, cols=cols, bit_min=bit_min, budget=budget)
    if kind == "exact":
        rows, cols = _size(rng, (32, 2048), (128, 11008), 512 * 11008, step)
        return dict(kind=kind, rows=rows, cols=cols, bit_min=bit_min)
    rows, cols = _size(rng, (64, 22016), (128, 22016), 22016 * 8192, step)
    return dict(kind=kind, rows=rows, cols=cols, bit_min=bit_min, budget=budget, scaled=scaled)


def _matrix(rows, cols, gen):
    W = torch.randn((rows, cols), generator=gen, device="cuda").mul_(0.02)
    at = torch.nonzero(torch.rand((rows * cols,), generator=gen, device="cuda") < 1e-3).view(-1)
    z = torch.randn((4, at.numel()), generator=gen, device="cuda")
    W.view(-1)[at] = 0.2 * z[0] / z[1:].square().mean(0).sqrt()        # Student's t with three degrees of freedom
    G = torch.randn((rows, cols), generator=gen, device="cuda").mul_(1.5).exp_()
    return W.half(), G


def _alpha(cols, gen):
    return torch.exp(0.25 * torch.randn((cols,), generator=gen, device="cuda"))


def _gram(cols, gen, samples=64):
    X = torch.randn((cols, samples), generator=gen, device="cuda")
    X += 0.3 * torch.randn((1, samples), generator=gen, device="cuda")
    X[torch.randperm(cols, generator=gen, device="cuda")[:4]] *= 8.0
    H = (X @ X.T / samples).half()
    upper = torch.triu(H)
    return upper + torch.triu(H, 1).T


def _packed_buffers(rows, cols, bits, pinned=False):
    kw = dict(pin_memory=True) if pinned else dict(device="cuda")
    return dict(packed=torch.zeros(Skim.packed_layout(rows, cols, bits)[1] // 4, dtype=torch.int32, **kw),
                row_order=torch.zeros(rows, dtype=torch.int32, **kw),
                group_info=torch.zeros(2 * (len(bits) + 1), dtype=torch.int64, **kw),
                lut=torch.zeros((rows, 1 << bits[-1]), dtype=torch.int16, **kw))


def prepare(case, seed):
    kind, rows, cols = case["kind"], case["rows"], case["cols"]
    bits = list(range(case["bit_min"], 5))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    W, G = _matrix(rows, cols, gen)
    ctx = Skim(device=0, rows=rows, cols=cols)
    st = dict(case, bits=bits, ctx=ctx, W=W, G=G)
    if kind == "pipeline":
        st["out"] = _packed_buffers(rows, cols, bits)
        st["alpha"] = _alpha(cols, gen) if case["scaled"] else None
    elif kind in ("alternate", "lfull_alternate"):
        st["alpha"] = _alpha(cols, gen)
        ctx.apply_scale(st["alpha"])
        cent, _, err = ctx.cluster_rows(W, G, bits, 10)
        st["row_bits"], _ = ctx.allocate_bits(err, bits, case["budget"])
        st["cent"] = cent
        if kind == "lfull_alternate":
            st["H"] = _gram(cols, gen)
    elif kind == "lfull_table":
        st["cent"], _, _ = ctx.cluster_rows(W, G, bits, 10)
        st["H"] = _gram(cols, gen)
        st["D"] = torch.empty((rows, cols), dtype=torch.float16, device="cuda")
        st["scratch"] = torch.empty(ctx.err_lfull_bytes(rows, cols), dtype=torch.uint8, device="cuda")
        st["table"] = torch.empty((rows, len(bits)), dtype=torch.float32, device="cuda")
    elif kind == "host":
        st["W"], st["G"] = W.cpu().pin_memory(), G.cpu().pin_memory()
        st["staging"] = torch.empty(Skim.host_staging_bytes(rows, cols, bits), dtype=torch.uint8, device="cuda")
        st["out"] = dict(_packed_buffers(rows, cols, bits, pinned=True),
                         err=torch.zeros((rows, len(bits)), dtype=torch.float32, pin_memory=True),
                         bits=torch.zeros(rows, dtype=torch.uint8, pin_memory=True))
    elif kind in ("dequantize", "matvec"):
        st["alpha"] = _alpha(cols, gen) if case["scaled"] else None
        ctx.apply_scale(st["alpha"])
        cent, _, err = ctx.cluster_rows(W, G, bits, 10)
        row_bits, _ = ctx.allocate_bits(err, bits, case["budget"])
        st["q"] = ctx.quantize(W, row_bits, cent, bits)
        st["W"] = st["G"] = None
        if kind == "matvec":
            st["x"] = torch.randn((cols,), generator=gen, device="cuda").half()
        else:
            st["out"] = torch.empty((rows, cols), dtype=torch.float16, device="cuda")
    return st


def run(st):
    kind, ctx, bits, W, G = st["kind"], st["ctx"], st["bits"], st["W"], st["G"]
    if kind == "pipeline":
        if st["alpha"] is not None:
            ctx.apply_scale(st["alpha"])
        cent, _, err = ctx.cluster_rows(W, G, bits, st["iters"])
        row_bits, total = ctx.allocate_bits(err, bits, st["budget"])
        q = ctx.quantize(W, row_bits, cent, bits, out=st["out"])
        return dict(q, cent=cent, err=err, row_bits=row_bits, total=total)
    if kind in ("alternate", "lfull_alternate"):
        alpha = st["alpha"].clone()                    # the update works in place
        ctx.apply_scale(alpha)
        cent, labels, err = ctx.cluster_rows_at(W, G, st["row_bits"], bits, st["iters"])
        if kind == "alternate":
            trace = ctx.scale_update(W, G, labels, alpha, steps=st["steps"])
        else:
            trace = ctx.scale_update_lfull(W, G, labels, alpha, st["H"], steps=st["steps"])
        return dict(cent=cent, labels=labels, err=err, alpha=alpha, trace=trace)
    if kind == "lfull_table":
        for k, b in enumerate(bits):
            ctx.residual(W, st["cent"], bits, width=b, out=st["D"])
            ctx.err_lfull(st["D"], st["H"], scratch=st["scratch"], out=st["table"][:, k], out_stride=len(bits))
        row_bits, total = ctx.allocate_bits(st["table"], bits, st["budget"])
        return dict(table=st["table"], residual=st["D"], row_bits=row_bits, total=total)
    if kind == "exact":
        cent, err = ctx.cluster_rows_exact(W, G, bits)
        return dict(cent=cent, err=err)
    if kind == "host":
        ctx.quantize_matrix_host(W, G, bits, st["iters"], st["budget"], st["staging"], st["out"])
        return st["out"]
    if kind == "dequantize":
        return ctx.dequantize(st["q"], st["cols"], bits, s=st["alpha"], out=st["out"])
    return ctx.matvec(st["q"], st["cols"], bits, st["x"], s=st["alpha"])


def work(case):
    """Bytes and operations of a pass.  Sorting, boundary searches and table lookups have no operation count that every
    implementation shares, so only the contractions and the per-element sums of the scaling update are counted."""
    kind, rows, cols = case["kind"], case["rows"], case["cols"]
    n = rows * cols
    widths = list(range(case["bit_min"], 5))
    sumk = sum(1 << b for b in widths)
    packed = n * case.get("budget", 0.0) / 8
    tables = rows * (4 * sumk + 4 * len(widths))                       # centroids and errors of every width
    emitted = packed + rows * (1 + 4 + 2 * 16)                         # codes, widths, row order, codebooks
    if kind in ("pipeline", "host"):
        return {"bytes": 6 * n + tables + emitted, "flops": 0}
    if kind == "alternate":
        # a step needs every weight, importance and label with the alpha that the step before it left
        return {"bytes": 7 * n + (7 * n + 4 * cols) * case["steps"] + rows * 4 * (sumk + 1), "flops": 16.0 * n * case["steps"]}
    if kind == "lfull_alternate":
        return {"bytes": 7 * n + (7 * n + 2 * cols * cols) * case["steps"], "flops": (2.0 * n * cols + 16.0 * n) * case["steps"]}
    if kind == "lfull_table":
        # the quadratic form of a symmetric H has rows * cols * (cols + 1) / 2 distinct products
        return {"bytes": 4 * n + 2 * cols * cols + tables, "flops": 1.0 * n * cols * len(widths)}
    if kind == "exact":
        return {"bytes": 6 * n + tables, "flops": 0}
    codebooks = packed + rows * (4 + 2 * 16) + 4 * cols * bool(case["scaled"])
    if kind == "dequantize":
        return {"bytes": codebooks + 2 * n, "flops": float(n)}
    return {"bytes": codebooks + 2 * cols + 4 * rows, "flops": 2.0 * n}


def tolerance(case):
    """Centroids, errors and alpha are binary32 results of binary64 sums; labels and codes may differ for elements at a
    midpoint.  The L-full update sums binary32 products of binary16 residuals, and 120 Adam steps carry that on."""
    kind = case["kind"]
    if kind == "lfull_alternate":
        return {"rel": 2e-4, "max": 2e-2, "differ": 1e-3}
    if kind == "dequantize":
        return {"rel": 1e-5, "max": 1e-3, "differ": 0.0}               # one binary16 rounding of a codebook entry
    return {"rel": 1e-5, "differ": 1e-3}
