"""The device NP with less scratch than it asks for."""
import numpy as np
import pytest

import oracle
import paper_2608_01907_gb300 as snap
from synth import initial_positions, tiny_graph

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [1, 2, 300])
def test_device_np_takes_fewer_blocks_when_its_scratch_is_refused(cuda, monkeypatch, count):
    """The third allocation is the scratch; a refusal is followed by a smaller
    request, except for a single sample, whose scratch is as small as it gets."""
    torch = cuda
    g = tiny_graph(900, 3000, seed=4)
    Y = initial_positions(g.n, 2)
    nodes = np.random.default_rng(1).integers(0, g.n, count).astype(np.int32)
    with snap.Layout(g.row_ptr, g.col_idx, opts=snap.make_options(keep_csr=True)) as L:
        pos = torch.from_numpy(Y).cuda()
        monkeypatch.setenv("SNAP_FAULT_INJECT", "alloc:3")
        if count == 1:
            with pytest.raises(snap.SnapError):
                L.neighborhood_preservation(pos, nodes)
            monkeypatch.delenv("SNAP_FAULT_INJECT")
        got, used = L.neighborhood_preservation(pos, nodes)
    ref = oracle.neighborhood_preservation(g.row_ptr, g.col_idx, g.n, Y.astype(np.float64), nodes)
    assert used == count
    assert abs(got - ref) < 1e-12
