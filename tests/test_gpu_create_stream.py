"""create waits for its stream: a handle may be used on any other one at once."""
import numpy as np
import pytest

import paper_2608_01907_gb300 as snap
from synth import edges_to_csr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sampler", [snap.SAMPLER_UNIFORM, snap.SAMPLER_DEGREE])
def test_create_of_a_synchronous_handle_leaves_nothing_under_way(cuda, sampler):
    """Large enough that a kernel launched after the last wait would still run
    when create returns."""
    torch = cuda
    n = 1_000_003
    v = np.arange(n)
    rp, ci = edges_to_csr(n, np.tile(v, 12), np.concatenate([(v + s) % n for s in range(1, 13)]))
    side = torch.cuda.Stream()
    opts = snap.make_options(mode=snap.MODE_SYNC, sampler=sampler)
    for _ in range(3):
        h = snap.snap_layout_create(rp, ci, None, n, opts, side)
        idle = side.query()
        side.synchronize()
        snap.snap_layout_destroy(h)
        assert idle
