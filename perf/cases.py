"""Performance cases: the calls a program that lays out graphs makes, from a
two-thousand-vertex graph to the 34M-edge R-MAT workload.

Every case refines a layout that already has its overall shape (positions
scattered around community centres) with the last epochs of a 30-epoch
schedule restarted at eta0 = 0.1.  An epoch costs the same at every step size;
small steps keep the lock-free modes' races from growing into different
layouts, so that two runs can be compared.  Graphs are
drawn on the GPU from the seed and handed to the library as host CSR arrays,
as its entry points take them.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2608_01907_gb300 as snap

TOTAL_EPOCHS = 30
ETA0 = 0.1
MODES = {"hogwild": snap.MODE_HOGWILD, "red": snap.MODE_HOGWILD_RED, "sync": snap.MODE_SYNC}
SAMPLERS = {"uniform": snap.SAMPLER_UNIFORM, "degree": snap.SAMPLER_DEGREE, "weights": snap.SAMPLER_WEIGHTS}


def _epochs(name, graph, n, edges, mode, k, epochs=1, sampler="uniform", substeps=1, cap=0.0):
    return dict(name=name, op="epochs", graph=graph, n=n, edges=edges, mode=mode, k=k, epochs=epochs,
                sampler=sampler, substeps=substeps, cap=cap)


def listed():
    return [
        # the 8-class graph of the paper's figures, the smallest graph laid out in earnest: a few
        # epochs in one call, where launches and the latency of one update count
        _epochs("sbm2k_red", "planted", 2_000, 22_557, "red", 3, epochs=3),
        # the Orkut-communities shape of the paper's teaser in the default mode
        _epochs("lfr260k_red", "powerlaw", 259_019, 6_893_156, "red", 3),
        # the benchmark's graph and mode: the largest ordinary job
        _epochs("rmat22_red", "rmat", 1 << 22, 34_000_000, "red", 3),
        # the racy-overwrite mode of the paper's lock-free scheme, more negatives than one random
        # block holds, sizes that divide by nothing
        _epochs("ragged_hogwild_k5", "powerlaw", 777_777, 9_999_991, "hogwild", 5),
        # degree-weighted negatives on a power-law graph
        _epochs("rmat20_degree", "rmat", 1 << 20, 8_000_000, "red", 3, sampler="degree"),
        # the deterministic mode as the benchmark runs it (16 chunks, capped steps)
        _epochs("rmat22_sync", "rmat", 1 << 22, 34_000_000, "sync", 3, substeps=16, cap=1.0),
        # the deterministic mode on a small graph: a few dozen short launches
        _epochs("sbm2k_sync", "planted", 2_000, 22_557, "sync", 3, substeps=4, cap=1.0),
        # many small graphs in one handle, epochs replayed as a CUDA graph
        dict(name="batch512", op="batch", count=512, nmin=100, nmax=20_000, mode="red", k=3, epochs=2),
        # one tick of the layout server: jobs of very different sizes in one launch
        dict(name="serve_tick", op="tick", count=24, emin=1_000, emax=2_000_000, mode="red", k=3),
        # the whole call from pinned host buffers: copy in, validate, build, a few epochs, copy out
        dict(name="run_lfr260k", op="run", graph="powerlaw", n=259_019, edges=6_893_156, mode="red", k=3, epochs=3),
        # quality report of a mid-size layout: neighbourhood preservation on sampled vertices
        dict(name="np_ragged", op="np", graph="powerlaw", n=1_000_003, edges=8_000_009, samples=256),
        # the exact objective, as the autotuner's gate and the quality tests evaluate it
        dict(name="objective_16k", op="objective", graph="planted", n=16_000, edges=120_000, exact=True, pairs=0,
             k=3, sampler="uniform"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["epochs", "epochs", "epochs", "epochs", "batch", "tick", "np", "objective", "run"])
    if op == "batch":
        return dict(op=op, count=_log_int(rng, 16, 512), nmin=rng.randint(60, 200),
                    nmax=_log_int(rng, 1_000, 20_000), mode=rng.choice(["red", "red", "hogwild"]),
                    k=rng.choice([1, 3, 3, 5]), epochs=rng.randint(1, 2))
    if op == "tick":
        return dict(op=op, count=rng.randint(2, 32), emin=rng.randint(500, 5_000),
                    emax=_log_int(rng, 100_000, 2_000_000), mode="red", k=rng.choice([1, 3, 3, 5]))
    graph = rng.choice(["planted", "powerlaw", "rmat"])
    n = _log_int(rng, 2_000, 2_000_000)
    edges = int(n * rng.uniform(4.0, 16.0))
    if op == "np":
        n = _log_int(rng, 2_000, 1_200_000)
        return dict(op=op, graph=graph, n=n, edges=int(n * rng.uniform(3.0, 10.0)), samples=rng.randint(64, 300))
    if op == "objective":
        exact = rng.random() < 0.6
        n = _log_int(rng, 1_000, 24_000) if exact else n
        return dict(op=op, graph=graph, n=n, edges=int(n * rng.uniform(4.0, 12.0)), exact=exact,
                    pairs=0 if exact else rng.randint(1 << 20, 1 << 24), k=rng.choice([1, 3, 5]),
                    sampler=rng.choice(["uniform", "uniform", "degree"]))
    if op == "run":
        # a whole call from host buffers: create, epochs, positions back
        return dict(op=op, graph=graph, n=n, edges=min(edges, 8_000_000), mode=rng.choice(["red", "sync"]), k=3,
                    epochs=rng.randint(1, 3))
    mode = rng.choice(["red", "red", "red", "hogwild", "sync"])
    k, epochs = rng.choice([1, 2, 3, 3, 4, 5, 10]), rng.randint(1, 2)
    sampler = rng.choice(["uniform", "uniform", "uniform", "degree", "weights"])
    edges = min(edges, (100_000_000 if sampler == "uniform" else 40_000_000) // ((1 + k) * epochs))
    case = _epochs("", graph, n, edges, mode, k, epochs=epochs, sampler=sampler,
                   substeps=rng.choice([1, 4, 16]) if mode == "sync" else 1,
                   cap=rng.choice([0.0, 1.0]) if mode == "sync" else 0.0)
    del case["name"]
    return case


# --------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _rand(g, m):
    return torch.rand(m, generator=g, device="cuda", dtype=torch.float64)


def _unique_keys(u, v, n):
    a, b = torch.minimum(u, v), torch.maximum(u, v)
    return torch.unique((a * n + b)[a != b])


def _exactly(sample, n, edges, g):
    """About `edges` distinct undirected edges from sample(m) -> (u, v), the surplus dropped at random."""
    keys = torch.empty(0, dtype=torch.int64, device="cuda")
    want = int(edges * 1.3) + 64
    for _ in range(6):
        keys = torch.unique(torch.cat([keys, _unique_keys(*sample(want), n)]))
        if keys.numel() >= edges:
            break
        want = 2 * (edges - keys.numel()) + int(0.2 * edges) + 64
    if keys.numel() > edges:
        keys = keys[torch.randperm(keys.numel(), generator=g, device="cuda")[:edges]]
    return keys


def _csr(keys, n):
    u, v = keys // n, keys % n
    both, _ = torch.sort(torch.cat([keys, v * n + u]))
    row_ptr = torch.searchsorted(both, torch.arange(n + 1, device="cuda", dtype=torch.int64) * n)
    return row_ptr, (both % n).to(torch.int32)


def _blocks(n, count):
    """Community of every vertex: `count` contiguous blocks of about n / count vertices."""
    return torch.arange(n, device="cuda", dtype=torch.int64) * count // n


def _planted(n, edges, g):
    comm = 8 if n < 20_000 else n // 2_000
    size = n // comm

    def sample(m):
        u = (_rand(g, m) * n).long()
        first = (u // size) * size
        v = torch.where(_rand(g, m) < 0.9, first + (_rand(g, m) * size).long(), (_rand(g, m) * n).long())
        return u, v.clamp(max=n - 1)
    return _exactly(sample, n, edges, g), _blocks(n, comm)


def _powerlaw(n, edges, g):
    """Power-law degrees (exponent 2.3) in communities, 10% of the edges across them."""
    comm = max(8, n // 3_000)
    label = _blocks(n, comm)
    w = (1.0 - _rand(g, n) * (1.0 - (4_000.0 / 10.0) ** -1.3)) ** (-1.0 / 1.3)
    cum = torch.cumsum(w, 0)
    last = torch.searchsorted(label, torch.arange(comm, device="cuda"), right=True) - 1
    end = cum[last]
    begin = torch.cat([torch.zeros(1, device="cuda", dtype=torch.float64), end[:-1]])

    def sample(m):
        u = torch.searchsorted(cum, _rand(g, m) * cum[-1]).clamp(max=n - 1)
        c = label[u]
        at = torch.where(_rand(g, m) < 0.9, begin[c] + _rand(g, m) * (end[c] - begin[c]), _rand(g, m) * cum[-1])
        return u, torch.searchsorted(cum, at).clamp(max=n - 1)
    return _exactly(sample, n, edges, g), label


def _rmat(n, edges, g):
    """R-MAT (a, b, c, d = .57, .19, .19, .05); a size that is no power of two folds the ids back."""
    scale = max(1, (n - 1).bit_length())

    def sample(m):
        u = torch.zeros(m, dtype=torch.int64, device="cuda")
        v = torch.zeros(m, dtype=torch.int64, device="cuda")
        for _ in range(scale):
            r = torch.rand(m, generator=g, device="cuda")
            u = (u << 1) | (r >= 0.76)
            v = (v << 1) | (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
        return u % n, v % n
    return _exactly(sample, n, edges, g), _blocks(n, 64)


def _positions(label, g):
    """A settled layout: vertices scattered around their communities' centres."""
    comm = int(label.max()) + 1
    centre = torch.randn(comm, 2, generator=g, device="cuda") * 3.0
    return (centre[label] + 0.6 * torch.randn(label.numel(), 2, generator=g, device="cuda")).contiguous()


def _graph(kind, n, edges, seed):
    """(row_ptr, col_idx, positions) on the device."""
    g = _generator(seed)
    keys, label = {"planted": _planted, "powerlaw": _powerlaw, "rmat": _rmat}[kind](n, edges, g)
    row_ptr, col = _csr(keys, n)
    return row_ptr, col, _positions(label, g)


def _batch_sizes(case):
    """(vertices, communities, edges drawn) of every graph: fixed by the case."""
    rng = random.Random(case["count"] * 1_000_003 + case["nmax"])
    return [(n, rng.randint(4, 32), int(n * rng.uniform(3.0, 10.0)))
            for n in (_log_int(rng, case["nmin"], case["nmax"]) for _ in range(case["count"]))]


def _batch_graph(case, seed):
    """Disjoint union of planted-partition graphs, drawn together."""
    g = _generator(seed)
    sizes = torch.tensor(_batch_sizes(case), dtype=torch.int64, device="cuda")
    ng, cg, mg = sizes[:, 0], sizes[:, 1], sizes[:, 2]
    offsets = torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), torch.cumsum(ng, 0)])
    total = int(offsets[-1])
    q = torch.repeat_interleave(torch.arange(ng.numel(), device="cuda"), mg)
    m = q.numel()
    block = (ng // cg).clamp(min=2)[q]
    u = (_rand(g, m) * ng[q]).long()
    inside = (u // block) * block + (_rand(g, m) * block).long()
    v = torch.where(_rand(g, m) < 0.9, torch.minimum(inside, ng[q] - 1), (_rand(g, m) * ng[q]).long())
    row_ptr, col = _csr(_unique_keys(offsets[q] + u, offsets[q] + v, total), total)
    which = torch.repeat_interleave(torch.arange(ng.numel(), device="cuda"), ng)
    local = torch.arange(total, device="cuda") - offsets[which]
    label = which * 32 + local * cg[which] // ng[which]
    return row_ptr, col, offsets, _positions(label, g)


def _job_sizes(case):
    """(kind, vertices, edges) of a tick's jobs: half R-MAT, half planted, edges log-uniform."""
    rng = random.Random(case["count"] * 1_000_003 + case["emax"])
    out = []
    for q in range(case["count"]):
        e = _log_int(rng, case["emin"], case["emax"])
        out.append(("rmat", 1 << max(6, math.ceil(math.log2(e / 4))), e) if q % 2 == 0
                   else ("planted", max(64, e // 5), e))
    return out


def _host(t):
    return np.ascontiguousarray(t.cpu().numpy())


def _pinned(t):
    return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)


def _node_weights(n, seed):
    """Caller weights of a weighted sampler: Pareto-like, some vertices never drawn."""
    rng = np.random.default_rng(seed)
    w = (rng.pareto(1.5, n) + 0.05).astype(np.float32)
    w[rng.random(n) < 0.1] = 0.0
    return w


def _options(case, seed, **more):
    sampler = case.get("sampler", "uniform")
    weights = _node_weights(case["n"], seed) if sampler == "weights" else None
    return snap.make_options(mode=MODES[case.get("mode", "red")], sampler=SAMPLERS[sampler], node_weights=weights,
                             sync_substeps=case.get("substeps", 1), sync_cap=case.get("cap", 0.0), **more)


def prepare(case, seed):
    """The handle a program keeps for its graph, and the positions it refines."""
    op = case["op"]
    schedule = snap.linear_schedule(ETA0, TOTAL_EPOCHS)
    state = dict(case=case, seed=seed, schedule=schedule)
    if op == "batch":
        row_ptr, col, offsets, pos = _batch_graph(case, seed)
        handle = snap.snap_layout_create_batch(_host(row_ptr), _host(col), _host(offsets.to(torch.int32)),
                                               _options(case, seed, cuda_graph=True))
        state.update(handle=_Handle(handle), pos=pos)
    elif op == "tick":
        jobs, kept = [], []
        for q, (kind, n, edges) in enumerate(_job_sizes(case)):
            row_ptr, col, pos = _graph(kind, n, edges, seed * 101 + q)
            layout = snap.Layout(_host(row_ptr), _host(col), opts=_options(case, seed))
            kept.append(layout)
            jobs.append((layout.handle, pos, 25 + q % 5, schedule, seed + q))
        state.update(layouts=kept, jobs=jobs, multi=snap.MultiEpoch(max_jobs=64))
    else:
        row_ptr, col, pos = _graph(case["graph"], case["n"], case["edges"], seed)
        if op == "run":
            state.update(row_ptr=_pinned(row_ptr).numpy(), col=_pinned(col).numpy(), pos=_pinned(pos),
                         opts=_options(case, seed), schedule=snap.linear_schedule(0.01, TOTAL_EPOCHS))
        else:
            opts = _options(case, seed, keep_csr=op == "np")
            state.update(layout=snap.Layout(_host(row_ptr), _host(col), opts=opts), pos=pos)
        if op == "np":
            state["nodes"] = _np_nodes(case, seed)
    return state


class _Handle:
    """Owns a batch handle."""

    def __init__(self, handle):
        self.handle = handle

    def __del__(self):
        snap.snap_layout_destroy(self.handle)


def _np_nodes(case, seed):
    return np.random.default_rng(seed).integers(0, case["n"], case["samples"]).astype(np.int32)


def run(state):
    case, pos, schedule, seed = state["case"], state.get("pos"), state["schedule"], state["seed"]
    op = case["op"]
    if op == "epochs":
        state["layout"].epochs(pos, TOTAL_EPOCHS - case["epochs"], case["epochs"], case["k"], schedule, seed)
        return pos
    if op == "batch":
        snap.snap_layout_epochs(state["handle"].handle, pos, TOTAL_EPOCHS - case["epochs"], case["epochs"],
                                case["k"], schedule, seed)
        return pos
    if op == "tick":
        state["multi"].epoch(state["jobs"], case["k"])
        return [job[1] for job in state["jobs"]]
    if op == "np":
        return state["layout"].neighborhood_preservation(pos, state["nodes"])
    if op == "objective":
        return state["layout"].objective(pos, case["k"], exact=case["exact"], pair_samples=case["pairs"], seed=seed)
    if op == "run":
        return snap.snap_layout_run(state["row_ptr"], state["col"], pos, case["epochs"], case["k"], schedule, seed,
                                    opts=state["opts"])
    raise ValueError(op)


def work(case):
    """One pass: the graph and the positions read once, the outputs written
    once; about 20 flops per attraction and per repulsion of a pair."""
    op = case["op"]
    if op == "batch":
        sizes = _batch_sizes(case)
        graphs = [(sum(s[0] for s in sizes), sum(s[2] for s in sizes))]
    elif op == "tick":
        graphs = [(n, e) for _, n, e in _job_sizes(case)]
    else:
        graphs = [(case["n"], case["edges"])]
    n, edges = sum(g[0] for g in graphs), sum(g[1] for g in graphs)
    stream = 8.0 * edges + 8.0 * n
    if op == "np":
        return {"bytes": stream + 8.0 * n, "flops": 5.0 * case["samples"] * n}
    if op == "objective":
        pairs = 0.5 * n * (n - 1) if case["exact"] else float(case["pairs"])
        return {"bytes": stream + 12.0 * n, "flops": 12.0 * pairs + 20.0 * edges}
    epochs = case.get("epochs", 1)
    return {"bytes": epochs * stream + 16.0 * n, "flops": epochs * 2.0 * edges * 20.0 * (1 + case["k"])}


# --------------------------------------------------------------------------
# What the deterministic calls return, in 64 bits
# --------------------------------------------------------------------------
_LOW = 0xFFFFFFFF


def _mul_hi_lo(const, x):
    """High and low 32 bits of const * x (x: int64 tensor of 32-bit values)."""
    low = (x & 0xFFFF) * const                  # < 2^48
    high = (x >> 16) * const + (low >> 16)      # < 2^49
    return high >> 16, ((high & 0xFFFF) << 16) | (low & 0xFFFF)


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors of 32-bit words."""
    k0, k1 = seed & _LOW, (seed >> 32) & _LOW
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & _LOW, (k1 + 0xBB67AE85) & _LOW
        hi0, lo0 = _mul_hi_lo(0xD2511F53, c0)
        hi1, lo1 = _mul_hi_lo(0xCD9E8D57, c2)
        c0, c1, c2, c3 = hi1 ^ c1 ^ k0, lo1, hi0 ^ c3 ^ k1, lo0
    return c0, c1, c2, c3


def _negative(word, src, n):
    u = (word * (n - 1)) >> 32
    return u + (u >= src).long()


def _attraction(d):
    return -0.1 * (1.0 + 8.0 / (1.0 + (d * d).sum(1, keepdim=True))) * d


def _repulsion(d):
    return d / (1.0 + (d * d).sum(1, keepdim=True)) ** 2


def _exact_sync_epoch(row_ptr, col, pos, case, seed, t, eta, eta0):
    """One synchronous epoch: per chunk of rows, the forces at the chunk's start summed, then one step."""
    n, nnz, parts, k, cap = pos.shape[0], col.numel(), case.get("substeps", 1), case["k"], case.get("cap", 0.0)
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), row_ptr[1:] - row_ptr[:-1])
    # chunk c starts at the first row that begins at or after c / parts of the edges
    want = torch.arange(parts + 1, device="cuda") * nnz
    first = row_ptr[torch.searchsorted(row_ptr * parts, want)].tolist()
    first[0], first[-1] = 0, nnz
    for b, e in zip(first[:-1], first[1:]):
        move = torch.zeros_like(pos)
        i, j = rows[b:e], col[b:e].long()
        edge = torch.arange(b, e, device="cuda")
        f = _attraction(pos[i] - pos[j])
        move.index_add_(0, i, f)
        move.index_add_(0, j, -f)
        zero = torch.zeros_like(edge)
        for m in range(k):
            if m % 4 == 0:
                words = _philox(edge & _LOW, edge >> 32, zero + t, zero + m // 4, seed)
            s = _negative(words[m % 4], i, n)
            f = _repulsion(pos[i] - pos[s])
            move.index_add_(0, i, f)
            move.index_add_(0, s, -f)
        step = eta * move
        if cap > 0:
            length = step.norm(dim=1, keepdim=True)
            limit = cap * eta / eta0
            step = torch.where(length > limit, step * (limit / length), step)
        pos = pos + step
    return pos


def _exact_sync(case, seed, begin, eta0):
    row_ptr, col, pos = _graph(case["graph"], case["n"], case["edges"], seed)
    pos = pos.double()
    for t in range(begin, begin + case["epochs"]):
        eta = max(eta0 * (1.0 - t / TOTAL_EPOCHS), eta0 * 1e-3)
        pos = _exact_sync_epoch(row_ptr, col, pos, case, seed, t, eta, eta0)
    return pos


def _exact_objective(case, seed):
    """Attraction over the edges and the weighted repulsion over the pairs (all, or the sampled ones)."""
    row_ptr, col, pos = _graph(case["graph"], case["n"], case["edges"], seed)
    n, pos = case["n"], pos.double()
    deg = (row_ptr[1:] - row_ptr[:-1]).double()
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), row_ptr[1:] - row_ptr[:-1])
    r2 = ((pos[rows] - pos[col.long()]) ** 2).sum(1)
    attr = float((0.1 * (0.5 * r2 + 4.0 * torch.log1p(r2))).sum()) / 2
    if case["exact"]:
        pairs = 0.0
        for b in range(0, n, 2_000):
            r2 = ((pos[b:b + 2_000, None] - pos[None]) ** 2).sum(2)
            u = (deg[b:b + 2_000, None] + deg[None]) * 0.5 / (1.0 + r2)
            pairs += float(u.sum()) - float(deg[b:b + 2_000].sum())
        pairs /= 2
    else:
        p = torch.arange(case["pairs"], device="cuda")
        words = _philox(p & _LOW, p >> 32, torch.full_like(p, 0xFFFFFFFD), torch.zeros_like(p), seed)
        i = (words[0] * n) >> 32
        j = _negative(words[1], i, n)
        u = (deg[i] + deg[j]) * 0.5 / (1.0 + ((pos[i] - pos[j]) ** 2).sum(1))
        pairs = float(u.sum()) / case["pairs"] * 0.5 * n * (n - 1)
    rep = case["k"] * pairs / (2.0 * (n - 1))
    return attr, rep, attr + rep


def _exact_np(case, seed):
    """Mean Jaccard index of each sample's two-hop set and as many nearest vertices (ties: smaller id)."""
    row_ptr, col, pos = _graph(case["graph"], case["n"], case["edges"], seed)
    n, pos = case["n"], pos.double()
    host_ptr = row_ptr.cpu().numpy()
    lengths = row_ptr[1:] - row_ptr[:-1]
    got = []
    for i in _np_nodes(case, seed).tolist():
        near = col[host_ptr[i]:host_ptr[i + 1]].long()
        if near.numel() == 0:
            continue
        count = lengths[near]
        base = torch.repeat_interleave(row_ptr[near] - torch.cumsum(count, 0) + count, count)
        member = torch.zeros(n, dtype=torch.bool, device="cuda")
        member[col[base + torch.arange(base.numel(), device="cuda")].long()] = True
        member[near] = True
        member[i] = False
        size = int(member.sum())
        d = ((pos - pos[i]) ** 2)
        d = d[:, 0] + d[:, 1]
        d[i] = math.inf
        both = int(member[torch.sort(d, stable=True).indices[:size]].sum())
        got.append(both / (2 * size - both))
    return (sum(got) / len(got) if got else 0.0), len(got)


def exact(case, seed):
    op = case["op"]
    if op == "np":
        return _exact_np(case, seed)
    if case.get("sampler", "uniform") != "uniform":
        return None   # the alias draws are the library's own
    if op == "objective":
        return _exact_objective(case, seed)
    if case.get("mode") == "sync":
        if op == "run":
            return _exact_sync(case, seed, 0, 0.01).cpu()
        return _exact_sync(case, seed, TOTAL_EPOCHS - case["epochs"], ETA0)
    return None   # the lock-free modes depend on the order of their races
