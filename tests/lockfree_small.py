"""Small lock-free workloads whose layouts are pinned (golden/lockfree_small.npz):
the last epochs of a settled layout, where small steps keep two runs close."""
from functools import lru_cache

import numpy as np
import torch

import paper_2608_01907_gb300 as snap
from synth import Graph, planted_partition_graph, rmat_graph, sbm_graph

EPOCHS = 30
PINNED = 1000

# graph, mode, sampler, negatives, epochs
CASES = {
    "sbm_red_k3": ("sbm", "red", "uniform", 3, 3),
    "rmat12_red_k3": ("rmat12", "red", "uniform", 3, 2),
    "rmat14_red_k5": ("rmat14", "red", "uniform", 5, 2),
    "rmat13_red_k2": ("rmat13", "red", "uniform", 2, 2),
    "rmat16_red_k1": ("rmat16", "red", "uniform", 1, 2),
    "rmat16_red_degree_k3": ("rmat16", "red", "degree", 3, 1),
    "sbm_red_degree_k3": ("sbm", "red", "degree", 3, 2),
    "rmat14_hogwild_k3": ("rmat14", "hogwild", "uniform", 3, 1),
    "batch_red_k3": ("batch", "red", "uniform", 3, 2),
    "tick_red_k5": ("tick", "red", "uniform", 5, 1),
}
_RMAT = {"rmat12": (12, 30_001), "rmat13": (13, 90_007), "rmat14": (14, 130_001), "rmat16": (16, 700_001)}


@lru_cache(maxsize=None)
def graph(kind):
    if kind == "sbm":
        return sbm_graph(n=2000, blocks=8, seed=4)
    if kind == "planted":
        return planted_partition_graph(12_001, 9, 16.0, 0.1, np.random.default_rng(8))
    scale, edges = _RMAT[kind]
    return rmat_graph(scale, edges, seed=6)


@lru_cache(maxsize=None)
def settled(kind):
    """Vertices scattered around the centres of 16 contiguous groups."""
    n = graph(kind).n
    rng = np.random.default_rng(n)
    centre = 3.0 * rng.standard_normal((16, 2))
    return (centre[np.arange(n) * 16 // n] + 0.6 * rng.standard_normal((n, 2))).astype(np.float32)


@lru_cache(maxsize=None)
def batch():
    """Disjoint union: (CSR of all, graph offsets, positions)."""
    kinds = ["sbm", "planted", "rmat12", "rmat13"]
    gs = [graph(k) for k in kinds]
    at = np.concatenate([[0], np.cumsum([g.n for g in gs])])
    ends = np.concatenate([[0], np.cumsum([g.nnz for g in gs])])
    row_ptr = np.concatenate([[0]] + [g.row_ptr[1:] + e for g, e in zip(gs, ends)])
    col = np.concatenate([g.col_idx + np.int32(a) for g, a in zip(gs, at)])
    whole = Graph(int(at[-1]), row_ptr.astype(np.int64), col.astype(np.int32))
    return whole, at.astype(np.int32), np.concatenate([settled(k) for k in kinds])


TICK = ["rmat12", "sbm", "rmat14", "planted", "rmat16"]


def run_case(name):
    """One run: the positions of all vertices, float64."""
    kind, mode, sampler, k, epochs = CASES[name]
    mode = snap.MODE_HOGWILD_RED if mode == "red" else snap.MODE_HOGWILD
    opts = snap.make_options(mode=mode, sampler=snap.SAMPLER_DEGREE if sampler == "degree" else snap.SAMPLER_UNIFORM)
    sched = snap.linear_schedule(0.1, EPOCHS)
    if kind == "tick":
        layouts = [snap.Layout(graph(q).row_ptr, graph(q).col_idx, opts=opts) for q in TICK]
        pos = [torch.from_numpy(settled(q).copy()).cuda() for q in TICK]
        multi = snap.MultiEpoch(max_jobs=len(TICK))
        multi.epoch([(h.handle, p, 25 + q, sched, 40 + q) for q, (h, p) in enumerate(zip(layouts, pos))], k)
        torch.cuda.synchronize()
        return np.concatenate([p.cpu().numpy() for p in pos]).astype(np.float64)
    if kind == "batch":
        g, offsets, y0 = batch()
        handle = snap.snap_layout_create_batch(g.row_ptr, g.col_idx, offsets, opts)
        pos = torch.from_numpy(y0.copy()).cuda()
        snap.snap_layout_epochs(handle, pos, EPOCHS - epochs, epochs, k, sched, 9)
        torch.cuda.synchronize()
        snap.snap_layout_destroy(handle)
    else:
        g = graph(kind)
        pos = torch.from_numpy(settled(kind).copy()).cuda()
        with snap.Layout(g.row_ptr, g.col_idx, opts=opts) as layout:
            layout.epochs(pos, EPOCHS - epochs, epochs, k, sched, 9)
            layout.check()
    return pos.cpu().numpy().astype(np.float64)


def pinned(name):
    """The PINNED vertices of highest degree (of the whole batch, or of all jobs)."""
    kind = CASES[name][0]
    if kind == "batch":
        deg = batch()[0].degrees
    elif kind == "tick":
        deg = np.concatenate([graph(q).degrees for q in TICK])
    else:
        deg = graph(kind).degrees
    return np.argsort(-deg, kind="stable")[:PINNED]
