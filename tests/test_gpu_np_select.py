"""The device NP's selection of the k nearest: graphs on both sides of its
size limits, layouts whose FP32 distances say little or nothing."""
import numpy as np
import pytest

import oracle
import paper_2608_01907_gb300 as snap
from synth import edges_to_csr

pytestmark = pytest.mark.gpu


def _graph(n, rng):
    """A ring with a few hubs, so that 2-hop sets range from 4 vertices to most of the graph."""
    ring = np.arange(n)
    hubs = rng.integers(0, n, 3)
    leaves = [rng.choice(n, n // d + 1, replace=False) for d in (2, 40, 500)]
    u = np.concatenate([ring] + [np.full(x.size, h) for h, x in zip(hubs, leaves)])
    v = np.concatenate([(ring + 1) % n] + leaves)
    return edges_to_csr(n, u, v), hubs, leaves


def _layout(kind, n, rng):
    if kind == "spread":
        return rng.standard_normal((n, 2))
    if kind == "clusters":      # distances over ten orders of magnitude
        return rng.choice([1e-4, 1.0, 1e6], (n, 1)) * rng.standard_normal((n, 2))
    if kind == "far":           # FP32 differences of a few ulps: FP64 agrees, most distances tie
        return 4096.0 + 1e-3 * rng.standard_normal((n, 2))
    if kind == "line":          # two distances in all
        return np.stack([np.arange(n) % 2, np.zeros(n)], axis=1)
    return np.full((n, 2), 0.25)   # "point": every distance is 0


@pytest.mark.parametrize("n,kinds", [(300, "spread line"), (8192, "spread point"), (8193, "spread clusters line"),
                                     (40_001, "spread far point"), (98_303, "clusters"), (98_305, "spread far"),
                                     (262_144, "spread"), (262_147, "spread line clusters")])
def test_device_np_equals_oracle_np_at_the_limits(cuda, n, kinds):
    torch = cuda
    rng = np.random.default_rng(n)
    (rp, ci), hubs, leaves = _graph(n, rng)
    nodes = np.concatenate([hubs, [x[0] for x in leaves], rng.integers(0, n, 6), [0, n - 1]]).astype(np.int32)
    with snap.Layout(rp, ci, opts=snap.make_options(keep_csr=True)) as L:
        for kind in kinds.split():
            Y = _layout(kind, n, rng).astype(np.float32)
            got, used = L.neighborhood_preservation(torch.from_numpy(Y).cuda(), nodes)
            ref = oracle.neighborhood_preservation(rp, ci, n, Y.astype(np.float64), nodes)
            assert used == nodes.size
            assert abs(got - ref) < 1e-12, kind
