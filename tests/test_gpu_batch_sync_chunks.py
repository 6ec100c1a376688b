"""Synchronous batches cut into chunks, with capped steps, and batches that run
past the end of their schedule."""
import numpy as np
import pytest

import paper_2608_01907_gb300 as snap
from gpu_helpers import gpu_layout
from synth import initial_positions, tiny_graph

pytestmark = pytest.mark.gpu

# every step size of this schedule is a short binary fraction, so the caps of a
# batch and of a graph alone round the same
SCHED = snap.linear_schedule(eta0=0.25, total_epochs=4)


def _copies(torch, g, B, opts, first, epochs, k, Y):
    """B copies of g as one batch, run from Y (B of them)."""
    rp, ci, offs = snap.batch_union([(g.row_ptr, g.col_idx)] * B)
    pos = torch.from_numpy(Y.copy()).cuda()
    h = snap.snap_layout_create_batch(rp, ci, offs, opts)
    try:
        for _ in range(2):   # the second call replays a captured graph
            pos.copy_(torch.from_numpy(Y))
            snap.snap_layout_epochs(h, pos, first, epochs, k, SCHED, 11)
            snap.snap_layout_check(h)
    finally:
        snap.snap_layout_destroy(h)
    return pos.cpu().numpy()


@pytest.mark.parametrize("sampler", [snap.SAMPLER_UNIFORM, snap.SAMPLER_DEGREE])
@pytest.mark.parametrize("B,S,k", [(3, 1, 3), (2, 2, 5), (4, 4, 1)])
def test_chunked_capped_batch_of_copies_equals_the_graph_alone(cuda, B, S, k, sampler):
    """B copies in B * S chunks are cut at the rows where the graph alone is
    cut into S, so every copy takes the same steps."""
    torch = cuda
    g = tiny_graph(403, 1501, seed=2)
    Y0 = np.concatenate([initial_positions(g.n, 5 + q) for q in range(B)])
    make = lambda parts: snap.make_options(mode=snap.MODE_SYNC, sync_substeps=parts, sync_cap=0.5, sampler=sampler)
    got = _copies(torch, g, B, make(B * S), 0, 4, k, Y0)
    for q in range(B):
        alone = gpu_layout(torch, g, Y0[q * g.n:(q + 1) * g.n], 4, k, SCHED, 11, opts=make(S))
        assert np.array_equal(got[q * g.n:(q + 1) * g.n].view(np.uint32), alone.view(np.uint32)), q


@pytest.mark.parametrize("replay", [False, True])
@pytest.mark.parametrize("mode", [snap.MODE_SYNC, snap.MODE_HOGWILD, snap.MODE_HOGWILD_RED])
def test_batch_past_its_schedule_stays_where_it_is(cuda, mode, replay):
    torch = cuda
    g = tiny_graph(203, 701, seed=3)
    Y0 = np.concatenate([initial_positions(g.n, 5 + q) for q in range(2)])
    opts = snap.make_options(mode=mode, cuda_graph=replay)
    past = _copies(torch, g, 2, opts, 4, 3, 3, Y0)
    assert np.array_equal(past.view(np.uint32), Y0.view(np.uint32))
    if mode == snap.MODE_SYNC:   # epochs 4 and 5 add nothing to the first four
        assert np.array_equal(_copies(torch, g, 2, opts, 0, 6, 3, Y0).view(np.uint32),
                              _copies(torch, g, 2, opts, 0, 4, 3, Y0).view(np.uint32))
