"""The clusterings that users of this library run, as measurable cases.

Each case is one pass through a public entry point: one matrix through
``Context.cluster`` (device, numpy or pinned host memory), one through
``lw_cluster_noalloc``, many matrices through a batch plan, or a burst of
requests through the serving loop.  A device matrix is consumed by a
clustering, so a pass on device memory first copies the matrix it clusters,
as a program that keeps its distances does.

Sizes and distributions: Gaussian mixtures (R^8 with 8 components, R^64 with
32 components of sigma U[0.5, 2], R^16 with 4 to 32 components), the same
with distances rounded to multiples of 1/1024 (many ties), and
conformer-like chains (128 beads, 64 seed chains, d = ||delta|| / sqrt(128)).
Distances are built on the GPU in FP32 from points drawn from the seed.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1709_06816_gb300 import Context, LINKAGES, autotune, native

DEVICE = "cuda:0"


# ---- the cases -------------------------------------------------------------

def listed():
    return [
        # the smallest call: a few dozen objects (an inner loop of a larger
        # program), all latency and launches
        {"name": "device_64_complete", "kind": "device", "n": 64, "linkage": "complete", "data": "gmm8"},
        # a small everyday clustering
        {"name": "device_512_complete", "kind": "device", "n": 512, "linkage": "complete", "data": "gmm8"},
        # protein conformations at their usual problem size
        {"name": "device_1968_complete", "kind": "device", "n": 1968, "linkage": "complete", "data": "conformer"},
        # numpy in, numpy out (a script that has its matrix on the host); odd size,
        # inversions
        {"name": "numpy_777_centroid", "kind": "numpy", "n": 777, "linkage": "centroid", "data": "gmm16"},
        # the entry point for callers that cannot allocate
        {"name": "noalloc_5003_average", "kind": "noalloc", "n": 5003, "linkage": "average", "data": "gmm16"},
        # a mid-sized matrix of odd size, Ward linkage
        {"name": "device_8191_ward", "kind": "device", "n": 8191, "linkage": "ward", "data": "gmm16"},
        # distances from a quantised source (many ties): single and average linkage
        {"name": "device_16384_single", "kind": "device", "n": 16384, "linkage": "single", "data": "gmm64q"},
        {"name": "device_16384_average", "kind": "device", "n": 16384, "linkage": "average", "data": "gmm64q"},
        # a pinned host matrix, host outputs: the matrix comes from another part
        # of the program through page-locked memory
        {"name": "pinned_12001_weighted", "kind": "pinned", "n": 12001, "linkage": "weighted", "data": "gmm16"},
        # the largest: a conformation study of 65536 chains
        {"name": "device_65536_complete", "kind": "device", "n": 65536, "linkage": "complete", "data": "conformer"},
        # thousands of independent clusterings of uneven size in one plan
        {"name": "batch_4096_jobs", "kind": "batch", "jobs": 4096, "n_lo": 64, "n_hi": 2048, "size_seed": 3},
        # a burst of requests of mixed size and linkage through the serving loop
        {"name": "serve_48_requests", "kind": "serve", "jobs": 48, "n_lo": 256, "n_hi": 32768, "size_seed": 4},
    ]


def _log_uniform(rng, lo, hi):
    return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng: random.Random):
    kind = rng.choices(["device", "numpy", "pinned", "noalloc", "batch", "serve"],
                       [6, 2, 2, 2, 2, 1])[0]
    if kind == "batch":
        hi = rng.choice([300, 700, 1500, 2048])
        return {"kind": kind, "jobs": _log_uniform(rng, 16, 2048), "n_lo": 64, "n_hi": hi,
                "size_seed": rng.randrange(1 << 30)}
    if kind == "serve":
        return {"kind": kind, "jobs": rng.randint(8, 40), "n_lo": 256, "n_hi": rng.randint(2000, 24000),
                "size_seed": rng.randrange(1 << 30)}
    linkage = rng.choice(list(LINKAGES))
    most = {"device": 32768, "numpy": 6000, "pinned": 16384, "noalloc": native.LW_NOALLOC_MAX_N}[kind]
    if linkage in ("single", "centroid"):
        most = min(most, 12000)  # many ties or inversions: few merges a round
    return {"kind": kind, "n": _log_uniform(rng, 64, most), "linkage": linkage,
            "data": rng.choice(["gmm8", "gmm16", "gmm64q", "conformer"])}


# ---- inputs ----------------------------------------------------------------

def _sizes(case):
    """(n, linkage) of every job of a batch or a burst: n log-uniform, linkage
    uniform over single, complete, average and Ward."""
    rng = random.Random(case["size_seed"])
    return [(_log_uniform(rng, case["n_lo"], case["n_hi"]), rng.randrange(4)) for _ in range(case["jobs"])]


def _points(gen, n, data):
    def uniform(lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(shape, generator=gen, device=DEVICE)

    def normal(*shape):
        return torch.randn(shape, generator=gen, device=DEVICE)

    if data == "conformer":
        steps = normal(64, 127, 3)
        steps = 3.8 * steps / steps.norm(dim=2, keepdim=True)
        chains = torch.cat([torch.zeros(64, 1, 3, device=DEVICE), steps.cumsum(dim=1)], dim=1).reshape(64, 384)
        chains -= chains.mean(dim=0)
        which = torch.randint(0, 64, (n,), generator=gen, device=DEVICE)
        return chains[which] + 0.5 * normal(n, 384)
    dim, parts = {"gmm8": (8, 8), "gmm16": (16, 16), "gmm64q": (64, 32)}[data]
    centers = uniform(-10.0, 10.0, parts, dim)
    sigma = uniform(0.5, 2.0, parts) if data == "gmm64q" else torch.ones(parts, device=DEVICE)
    which = torch.randint(0, parts, (n,), generator=gen, device=DEVICE)
    return centers[which] + sigma[which, None] * normal(n, dim)


def _packed(points, data, out):
    """The strict upper triangle of the distances, row by row, into `out`."""
    n = points.shape[0]
    block = max(1, min(n, (1 << 27) // n))
    at = 0
    for r in range(0, n - 1, block):
        rows = points[r:min(r + block, n - 1)]
        d = torch.cdist(rows, points[r:])
        if data == "conformer":
            d = d / math.sqrt(128.0)
        elif data == "gmm64q":
            d = torch.round(d * 1024.0) / 1024.0
        keep = torch.ones(d.shape, dtype=torch.bool, device=DEVICE).triu(diagonal=1)
        part = torch.masked_select(d, keep)
        out[at:at + part.numel()] = part
        at += part.numel()
    return out


def _matrix(seed, n, data):
    gen = torch.Generator(DEVICE)
    gen.manual_seed(seed)
    return _packed(_points(gen, n, data), data, torch.empty(n * (n - 1) // 2, device=DEVICE))


class _Plan:
    """A batch plan and the buffers its jobs point to."""

    def __init__(self, ctx, work, sizes):
        self.ctx = ctx
        self.sizes = sizes
        steps = sum(n - 1 for n, _ in sizes)
        self.merges = torch.empty((steps, 2), dtype=torch.int32, device=DEVICE)
        self.heights = torch.empty(steps, dtype=torch.float32, device=DEVICE)
        self.jobs = (native.LwJob * len(sizes))()
        cell = step = 0
        for job, (n, linkage) in zip(self.jobs, sizes):
            job.dist = work.data_ptr() + 4 * cell
            job.n = n
            job.linkage = linkage
            job.status = -1
            job.merges_out = self.merges.data_ptr() + 8 * step
            job.heights_out = self.heights.data_ptr() + 4 * step
            cell += n * (n - 1) // 2
            step += n - 1
        self.handle = native.lw_batch_create(ctx.handle, self.jobs)

    def __del__(self):
        if getattr(self, "handle", None):
            native.lw_batch_destroy(self.handle)
            self.handle = None


def _many(case, seed):
    """The matrices of a batch or a burst, one after another in one buffer."""
    sizes = _sizes(case)
    cells = torch.empty(sum(n * (n - 1) // 2 for n, _ in sizes), device=DEVICE)
    gen = torch.Generator(DEVICE)
    gen.manual_seed(seed)
    parts = []
    at = 0
    for n, _ in sizes:
        m = n * (n - 1) // 2
        parts.append(_packed(_points(gen, n, "gmm16"), "gmm16", cells[at:at + m]))
        at += m
    return sizes, cells, parts


def prepare(case, seed):
    kind = case["kind"]
    state = {"kind": kind}
    if kind == "batch":
        sizes, cells, _ = _many(case, seed)
        stream = torch.cuda.Stream(DEVICE)
        ctx = Context(0, stream)
        autotune.apply(ctx)
        work = torch.empty_like(cells)
        state.update(cells=cells, work=work, stream=stream, plan=_Plan(ctx, work, sizes))
    elif kind == "serve":
        sizes, cells, parts = _many(case, seed)
        steps = sum(n - 1 for n, _ in sizes)
        state.update(sizes=sizes, cells=cells, parts=parts,
                     server=native.Server(0, budget_bytes=16 << 30, lanes=48),
                     merges=torch.empty((steps, 2), dtype=torch.int32, device=DEVICE),
                     heights=torch.empty(steps, dtype=torch.float32, device=DEVICE))
    else:
        n = case["n"]
        D = _matrix(seed, n, case["data"])
        state.update(n=n, linkage=case["linkage"])
        if kind == "numpy":
            state.update(D=D.cpu().numpy(), ctx=Context(0))
        elif kind == "pinned":
            state.update(D=D.cpu().pin_memory(), ctx=Context(0))
        elif kind == "noalloc":
            state.update(D=D, work=torch.empty_like(D), stream=torch.cuda.Stream(DEVICE),
                         merges=torch.empty((n - 1, 2), dtype=torch.int32, device=DEVICE),
                         heights=torch.empty(n - 1, dtype=torch.float32, device=DEVICE))
        else:
            stream = torch.cuda.Stream(DEVICE)
            state.update(D=D, work=torch.empty_like(D), stream=stream, ctx=Context(0, stream))
    torch.cuda.synchronize()
    return state


# ---- one pass --------------------------------------------------------------

def run(state):
    kind = state["kind"]
    if kind == "batch":
        plan = state["plan"]
        with torch.cuda.stream(state["stream"]):
            state["work"].copy_(state["cells"])
        native.lw_batch_run(plan.handle, plan.ctx.handle)
        if native.lw_batch_wait(plan.handle, plan.jobs) != 0:
            raise RuntimeError("a job of the batch failed")
        return plan.merges, plan.heights
    if kind == "serve":
        server, step = state["server"], 0
        for part, (n, linkage) in zip(state["parts"], state["sizes"]):
            server.submit(part, n, linkage, state["merges"][step:step + n - 1],
                          state["heights"][step:step + n - 1])
            step += n - 1
        if server.drain() != 0:
            raise RuntimeError("a request failed")
        return state["merges"], state["heights"]
    n = state["n"]
    if kind in ("numpy", "pinned"):
        return state["ctx"].cluster(state["D"], n, state["linkage"])
    with torch.cuda.stream(state["stream"]):
        state["work"].copy_(state["D"])
        if kind == "noalloc":
            native.lw_cluster_noalloc(state["work"], n, LINKAGES[state["linkage"]], state["merges"],
                                      state["heights"], state["stream"])
            return state["merges"], state["heights"]
        return state["ctx"].cluster(state["work"], n, state["linkage"])


# ---- what a pass cannot do without ------------------------------------------

def work(case):
    """Bytes: every distance read once, every merge (two int32) and height
    (float) written once.  Operations: n(n-1)/2 - (n-1) cells are recomputed
    per clustering (one for every live cluster beside the merged two), eight
    each (four products, three sums, one difference; the absolute value and
    the coefficients are not counted)."""
    sizes = [n for n, _ in _sizes(case)] if "jobs" in case else [case["n"]]
    return {"bytes": sum(2 * n * (n - 1) + 12 * (n - 1) for n in sizes),
            "flops": sum(8 * (n - 1) * (n - 2) // 2 for n in sizes)}


# ---- the same in 64 bits ----------------------------------------------------

def exact(case, seed):
    """The heights of the step-by-step iteration in FP64 (lowest row, then
    lowest column among equal distances); the merges are whole numbers."""
    if "jobs" in case or case["n"] > 16384:
        return None
    n, linkage = case["n"], case["linkage"]
    D = torch.full((n, n), math.inf, dtype=torch.float64, device=DEVICE)
    r, c = torch.triu_indices(n, n, 1, device=DEVICE)
    D[r, c] = _matrix(seed, n, case["data"]).double()
    D[c, r] = D[r, c]
    size = torch.ones(n, dtype=torch.float64, device=DEVICE)
    heights = np.empty(n - 1)
    for t in range(n - 1):
        low = D.min(dim=1).values
        h = low.min()
        i = int((low == h).nonzero()[0, 0])
        j = int((D[i] == h).nonzero()[0, 0])
        dij = float(h)
        heights[t] = dij
        a, b = D[i].clone(), D[j].clone()
        ni, nj = float(size[i]), float(size[j])
        if linkage == "single":
            new = torch.minimum(a, b)
        elif linkage == "complete":
            new = torch.maximum(a, b)
        elif linkage == "average":
            new = (ni * a + nj * b) / (ni + nj)
        elif linkage == "weighted":
            new = 0.5 * a + 0.5 * b
        elif linkage == "centroid":
            new = (ni * a + nj * b) / (ni + nj) - ni * nj / (ni + nj) ** 2 * dij
        else:
            total = ni + nj + size
            new = ((ni + size) * a + (nj + size) * b - size * dij) / total
        gone = torch.isinf(a) | torch.isinf(b)  # retired slots, i and j themselves
        new = torch.where(gone, math.inf, new)
        D[i], D[:, i] = new, new
        D[j], D[:, j] = math.inf, math.inf
        size[i] += nj
    if case["kind"] not in ("numpy", "pinned"):
        return None, torch.from_numpy(heights)
    return None, heights
