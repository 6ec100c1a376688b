"""The device NP on layouts whose squared distances leave the range of FP32:
they are infinite there, and the FP64 distances decide all the same."""
import numpy as np
import pytest

import oracle
import paper_2608_01907_gb300 as snap
from synth import edges_to_csr

pytestmark = pytest.mark.gpu


def _graph(n, rng):
    """A ring with two hubs: 2-hop sets from 4 vertices to half of the graph."""
    ring = np.arange(n)
    hubs = rng.integers(0, n, 2)
    leaves = [rng.choice(n, n // d + 1, replace=False) for d in (2, 50)]
    u = np.concatenate([ring] + [np.full(x.size, h) for h, x in zip(hubs, leaves)])
    v = np.concatenate([(ring + 1) % n] + leaves)
    return edges_to_csr(n, u, v), hubs


def _layout(kind, n, rng):
    y = rng.standard_normal((n, 2))
    if kind == "wide":          # every squared distance overflows
        return 1e20 * y
    if kind == "mixed":         # some do
        return rng.choice([1.0, 1e18, 1e22], (n, 1)) * y
    if kind == "edge":          # around the largest float
        return 1.3e19 * y
    return 3e38 * np.clip(y, -1.0, 1.0)   # "largest": differences overflow as well


@pytest.mark.parametrize("kind", ["wide", "mixed", "edge", "largest"])
@pytest.mark.parametrize("n", [300, 8192, 40_001, 262_147])   # the whole graph in the candidate list, or a bracket
def test_device_np_of_wide_layouts_equals_the_oracles(cuda, n, kind):
    torch = cuda
    rng = np.random.default_rng(n)
    (rp, ci), hubs = _graph(n, rng)
    nodes = np.concatenate([hubs, rng.integers(0, n, 8), [0, n - 1]]).astype(np.int32)
    Y = _layout(kind, n, rng).astype(np.float32)
    with snap.Layout(rp, ci, opts=snap.make_options(keep_csr=True)) as L:
        got, used = L.neighborhood_preservation(torch.from_numpy(Y).cuda(), nodes)
    ref = oracle.neighborhood_preservation(rp, ci, n, Y.astype(np.float64), nodes)
    assert used == nodes.size
    assert abs(got - ref) < 1e-12
