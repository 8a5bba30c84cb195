"""The workloads this framework is timed on: barcodes of point clouds through
the calls a program makes (ph0.barcodes, ph0.barcodes_early, ph0.death_values
and ph0.Batch with their backward passes, ph0.h1, serve.Server), from the
smallest clouds, where launches count, to the largest, where the edges do.

A case is a dict of plain values.  kind:
  bars     one cloud, ph0.barcodes
  early    one cloud, ph0.barcodes_early
  grad     one cloud, ph0.death_values, loss sum(death^2), backward
  batch    `count` clouds of one shape, ph0.Batch.death_values, the same loss
           summed over the clouds, backward
  h1       one cloud, ph0.h1
  stream   `count` clouds of mixed sizes through one serve.Server, all queued
           at once, until the last result is back
cloud: uniform (the unit cube), mixture (8 Gaussians), circles (4 noisy unit
circles, one after the other); inputs.py draws them.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2203_02527_gb300 import inputs, ph0, serve


def listed():
    return [
        # the paper's small experiments (N = 50..700): one cloud at a time, launch-bound
        {"name": "bars_uniform_256x3", "kind": "bars", "cloud": "uniform", "n": 256, "d": 3},
        # the paper's largest cloud, in its unit square
        {"name": "bars_uniform_700x2", "kind": "bars", "cloud": "uniform", "n": 700, "d": 2},
        # a clustered cloud of a few thousand points: the everyday single call
        {"name": "bars_mixture_4096x3", "kind": "bars", "cloud": "mixture", "n": 4096, "d": 3},
        # embedding vectors: a ragged size and a dimension without an instance of its own
        {"name": "bars_mixture_9001x24", "kind": "bars", "cloud": "mixture", "n": 9001, "d": 24},
        # the benchmark cloud: 537M edges
        {"name": "bars_circles_32768x16", "kind": "bars", "cloud": "circles", "n": 32768, "d": 16},
        # a large planar cloud: 1.25G edges, the sort and the reduction far above the distances
        {"name": "bars_uniform_50021x2", "kind": "bars", "cloud": "uniform", "n": 50021, "d": 2},
        # the early-terminating call on a large cloud in space
        {"name": "early_uniform_20011x3", "kind": "early", "cloud": "uniform", "n": 20011, "d": 3},
        # one topological-loss term of a training step: deaths and their gradient
        {"name": "grad_mixture_1500x8", "kind": "grad", "cloud": "mixture", "n": 1500, "d": 8},
        # the descent workload: 64 clouds a step, forward and backward
        {"name": "batch_uniform_64x2048x3", "kind": "batch", "cloud": "uniform", "count": 64, "n": 2048, "d": 3},
        # first homology of the paper's largest cloud
        {"name": "h1_uniform_700x2", "kind": "h1", "cloud": "uniform", "n": 700, "d": 2},
        # serving: clouds of 64 to 8192 points in 2 to 32 dimensions, all queued at once
        {"name": "stream_128", "kind": "stream", "count": 128, "n": 8192, "d": 32},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["bars", "bars", "bars", "early", "grad", "batch", "h1", "stream"])
    d = rng.choice([1, 2, 3, 4, 5, 8, 13, 16, 24, 32])
    cloud = rng.choice(["uniform", "mixture", "circles"] if d >= 2 else ["uniform", "mixture"])
    # per edge the cost is a constant and a share that grows with the
    # dimension: the most points whose cost stays below the largest listed case
    n_max = int(50000 * math.sqrt(1.0 / (1.0 + d / 8.0)))
    if kind == "bars":
        n = _log_uniform(rng, 64, n_max)
    elif kind == "early":
        n = _log_uniform(rng, 2000, n_max)
    elif kind == "grad":
        n = _log_uniform(rng, 64, 8192)
    elif kind == "h1":
        d = rng.choice([2, 3, 8])
        cloud = rng.choice(["uniform", "mixture"])
        n = _log_uniform(rng, 50, 800)
    else:
        n = _log_uniform(rng, 100, 3000)
    case = {"kind": kind, "cloud": cloud, "n": n, "d": d}
    if kind == "batch":
        case["count"] = rng.randint(2, 64)
    if kind == "stream":
        case = {"kind": kind, "count": rng.randint(16, 128), "n": 8192, "d": 32}
    return case


def _cloud(case, seed):
    n, d = case["n"], case["d"]
    if case["cloud"] == "uniform":
        return inputs.uniform(n, d, seed=seed)
    if case["cloud"] == "mixture":
        return inputs.gaussian_mixture(n, d, k=8, sigma=0.05, center_range=10.0, seed=seed)
    return inputs.noisy_circles((n + 3) // 4, 4, d, seed=seed)[:n]


def _clouds(case, seed):
    if case["kind"] == "stream":
        rng = np.random.Generator(np.random.PCG64(seed))
        return [inputs.gaussian_mixture(n, d, k=int(rng.integers(1, 17)), sigma=float(rng.uniform(0.05, 0.5)),
                                        seed=seed * 1000 + i) for i, (n, d) in enumerate(_stream_shapes(case))]
    if case["kind"] == "batch":
        return [_cloud(case, seed * 1000 + i) for i in range(case["count"])]
    return [_cloud(case, seed)]


_server = None


def _serving_context():
    """The serving context of this process (a program keeps one)."""
    global _server
    if _server is None:
        _server = serve.Server(mem_budget=8 << 30, host_budget=1 << 30, streams=4)
    return _server


def prepare(case, seed):
    clouds = _clouds(case, seed)
    state = {"kind": case["kind"]}
    if case["kind"] == "stream":
        state["clouds"] = clouds
        state["server"] = _serving_context()
        return state
    pts = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in clouds]
    if case["kind"] in ("grad", "batch"):
        pts = [p.requires_grad_(True) for p in pts]
    state["pts"] = pts
    if case["kind"] == "batch":
        state["batch"] = ph0.Batch([tuple(p.shape) for p in pts])
    return state


def _bars(b):
    return {"death": b.death, "raw": b.raw, "inf": b.inf_raw}


def run(state):
    kind = state["kind"]
    if kind == "stream":
        clouds = state["clouds"]
        done = serve.run_stream(state["server"], clouds)
        bars = np.concatenate([done[i].bars for i in range(len(clouds))])
        return {"death": bars["death"].copy(), "raw": bars.view(np.uint8),
                "status": np.array([done[i].status for i in range(len(clouds))]),
                "inf_vertex": np.array([done[i].inf_vertex for i in range(len(clouds))])}
    pts = state["pts"]
    if kind == "bars":
        b = ph0.barcodes(pts[0])
        return {**_bars(b), "n_distinct": b.stats["n_distinct"], "n_bars": b.stats["n_bars"]}
    if kind == "early":
        return _bars(ph0.barcodes_early(pts[0]))
    if kind == "h1":
        bars, stats = ph0.h1(pts[0])
        return {"raw": bars.view(np.uint8), "birth_sq": bars["birth_sq"].copy(), "death_sq": bars["death_sq"].copy(),
                "n_bars": stats["n_bars"], "n_triangles": stats["n_triangles"]}
    if kind == "grad":
        deaths = [ph0.death_values(pts[0])]
    else:
        deaths = list(state["batch"].death_values(pts))
    loss = sum((dv ** 2).sum() for dv in deaths)
    grads = torch.autograd.grad(loss, pts)
    return {"loss": loss.detach(), "deaths": torch.stack([dv.detach() for dv in deaths]), "grads": torch.stack(grads)}


def work(case):
    """Bytes: the points read once, the results written once.  Operations: the
    3d - 1 binary64 operations of each pair's squared distance (first homology:
    one look at each triangle's three edges beside them)."""
    if case["kind"] == "stream":
        shapes = _stream_shapes(case)
    else:
        shapes = [(case["n"], case["d"])] * case.get("count", 1)
    nbytes = flops = 0.0
    for n, d in shapes:
        m = n * (n - 1) / 2
        nbytes += 4.0 * n * d
        flops += m * (3 * d - 1)
        if case["kind"] == "h1":
            nbytes += 72.0 * (m - (n - 1))
            flops += 3.0 * n * (n - 1) * (n - 2) / 6
        elif case["kind"] in ("grad", "batch"):
            nbytes += 8.0 * (n - 1) + 4.0 * n * d  # deaths, gradient
        else:
            nbytes += 40.0 * (n - 1)
    return {"bytes": nbytes, "flops": flops}


def _stream_shapes(case):
    # sizes spread evenly over their logarithm, the four dimensions in turn,
    # arriving in an order that depends on the case alone
    k = case["count"]
    shapes = [(int(64 * 128 ** ((i + 0.5) / k)), (2, 3, 8, 32)[i % 4]) for i in range(k)]
    random.Random(k).shuffle(shapes)
    return shapes


def _spanning_trees(x):
    """Minimum spanning trees of a batch of clouds ([c, n, d] binary64) by
    Prim's rule: lengths [c, n-1] in increasing order and the edges' endpoints
    (u, v), [c, n-1] each in the same order."""
    c, n, _ = x.shape
    rows = torch.arange(c, device=x.device)
    inside = torch.zeros((c, n), dtype=torch.bool, device=x.device)
    best = torch.full((c, n), math.inf, dtype=torch.float64, device=x.device)
    link = torch.zeros((c, n), dtype=torch.long, device=x.device)
    new = torch.zeros(c, dtype=torch.long, device=x.device)
    length, us, vs = [], [], []
    for _ in range(n - 1):
        inside[rows, new] = True
        best[rows, new] = math.inf
        d2 = ((x - x[rows, new].unsqueeze(1)) ** 2).sum(-1)
        closer = (d2 < best) & ~inside
        best = torch.where(closer, d2, best)
        link = torch.where(closer, new.unsqueeze(1), link)
        w, new = best.min(1)
        length.append(w)
        us.append(link[rows, new])
        vs.append(new)
    w, u, v = torch.stack(length, 1), torch.stack(us, 1), torch.stack(vs, 1)
    w, order = w.sort(1)
    return w.sqrt(), u.gather(1, order), v.gather(1, order)


def exact(case, seed):
    """Deaths are the lengths of the minimum spanning tree; the gradient of
    the sum of their squares is 2 (x_u - x_v) at u and its negative at v."""
    if case["kind"] == "h1":
        return None
    clouds = _clouds(case, seed)
    if case["kind"] == "stream":
        if sum(len(x) for x in clouds) > 300000:
            return None
        out = []
        for x in clouds:
            w, _, _ = _spanning_trees(torch.from_numpy(x).cuda().double().unsqueeze(0))
            out.append(w[0].cpu().numpy())
        return {"death": np.concatenate(out), "raw": None, "status": None, "inf_vertex": None}
    x = torch.from_numpy(np.stack(clouds)).cuda().double()
    w, u, v = _spanning_trees(x)
    if case["kind"] == "bars":
        return {"death": w[0], "raw": None, "inf": None, "n_distinct": None, "n_bars": None}
    if case["kind"] == "early":
        return {"death": w[0], "raw": None, "inf": None}
    rows = torch.arange(x.shape[0], device=x.device).unsqueeze(1)
    step = 2.0 * (x[rows, u] - x[rows, v])
    grad = torch.zeros_like(x)
    for i in range(x.shape[0]):
        grad[i].index_add_(0, u[i], step[i])
        grad[i].index_add_(0, v[i], -step[i])
    return {"loss": (w ** 2).sum(), "deaths": w, "grads": grad}
