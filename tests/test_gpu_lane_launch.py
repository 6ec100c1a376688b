"""Lock-free launches of every width: how many lanes, how many of them to a
warp, short last chunks and slot groups.  On a perfect matching the order of
the entries does not matter, so the outcome is known."""
import numpy as np
import pytest

import oracle
import paper_2608_01907_gb300 as snap
from gpu_helpers import SYNC_RTOL, gpu_layout, parity_error, schedule_dict
from synth import Graph, edges_to_csr, initial_positions

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 5, 127, 129, 1000, 4099, 60_001]


def _matching(m):
    """m edges without a common vertex, ends far apart."""
    n = 2 * m
    return Graph(n, *edges_to_csr(n, np.arange(m), n - 1 - np.arange(m)))


@pytest.mark.parametrize("mode", [snap.MODE_HOGWILD, snap.MODE_HOGWILD_RED])
@pytest.mark.parametrize("m", SIZES)
def test_matching_without_negatives_equals_algorithm1(cuda, mode, m):
    """k = 0: an edge's two steps touch only its own ends, so any number of
    lanes gives Algorithm 1's positions."""
    g = _matching(m)
    Y0 = initial_positions(g.n, 3)
    sched = snap.linear_schedule(eta0=0.5, total_epochs=4)
    ref = oracle.seq(g.row_ptr, g.col_idx, g.n, Y0, 2, 0, schedule_dict(sched), seed=5)
    for block, share, seg in ((0, 0.0, 0), (32, 0.0, 0), (0, 1.0, 8), (0, 0.05, 4096)):
        opts = snap.make_options(mode=mode, block_threads=block, max_inflight=share, segment_edges=seg)
        got = gpu_layout(cuda, g, Y0, 2, 0, sched, seed=5, opts=opts)
        assert parity_error(got, ref) < SYNC_RTOL


@pytest.mark.parametrize("sampler", [snap.SAMPLER_UNIFORM, snap.SAMPLER_DEGREE])
@pytest.mark.parametrize("m,k", [(2, 1), (127, 3), (1000, 3), (4099, 5), (60_001, 3), (60_001, 2)])
def test_matching_with_negatives_moves_by_the_summed_forces(cuda, sampler, m, k):
    """With steps of 1e-3 every vertex moves by 1e-3 times the sum of its
    forces at the start, up to the change of those forces along its own and
    its partners' updates (about 2 + 2k of them, each moving a vertex by at
    most 1e-3 times a force below 1): below 0.05 of a unit force.  An entry
    taken twice or not at all would change the sum by its whole attraction."""
    g = _matching(m)
    Y0 = initial_positions(g.n, 3)
    sched = snap.linear_schedule(eta0=1e-3, total_epochs=1)
    sampling = oracle.Sampler.degree(g.row_ptr) if sampler == snap.SAMPLER_DEGREE else None
    want = oracle.epoch_displacement(g.row_ptr, g.col_idx, g.n, Y0, 0, k, 9, sampler=sampling)
    got = gpu_layout(cuda, g, Y0, 1, k, sched, seed=9, opts=snap.make_options(sampler=sampler))
    moved = (got.astype(np.float64) - Y0) / 1e-3
    assert np.abs(moved - want).max() < 0.05
