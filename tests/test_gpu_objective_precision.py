"""The attraction sum keeps its precision whatever the length of the chunks."""
import numpy as np
import pytest

import paper_2608_01907_gb300 as snap
from synth import edges_to_csr

pytestmark = pytest.mark.gpu

# terms within 16 x 2^-24, summed in FP32 over at most 32 edges, then in FP64
RTOL = (32 + 16) * 2.0 ** -24


@pytest.mark.parametrize("keep", [False, True])
@pytest.mark.parametrize("seg", [0, 12, 4096])
def test_attraction_of_equal_edges(cuda, seg, keep):
    """A ring whose edges all have length d: equal terms round the same way
    every time they are added, so a long FP32 sum drifts."""
    torch = cuda
    n = 12_290
    rp, ci = edges_to_csr(n, np.arange(n), (np.arange(n) + 1) % n)
    with snap.Layout(rp, ci, opts=snap.make_options(segment_edges=seg, keep_csr=keep)) as L:
        for d in np.float32([0.7, 1.0, 1.3, 2.1, 3.3]):
            Y = np.stack([d * (np.arange(n) % 2), np.zeros(n)], axis=1).astype(np.float32)
            attr, _, _ = L.objective(torch.from_numpy(Y).cuda(), 0)
            r2 = float(d) ** 2
            assert attr == pytest.approx(n * 0.1 * (0.5 * r2 + 4.0 * np.log1p(r2)), rel=RTOL)
