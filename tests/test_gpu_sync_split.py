"""The synchronous epoch's split of a chunk over lanes, and the edges whose
two copies lie in one chunk (their forces are added by each row for itself)."""
import numpy as np
import pytest

import oracle
import paper_2608_01907_gb300 as snap
from gpu_helpers import SYNC_RTOL, gpu_layout, parity_error, schedule_dict
from synth import Graph, edges_to_csr, initial_positions, tiny_graph

pytestmark = pytest.mark.gpu


def _graph(name):
    if name == "star":        # one row holds half of the edges; with chunks, most copies lie in different ones
        n = 130
        return Graph(n, *edges_to_csr(n, np.zeros(n - 1, np.int64), np.arange(1, n)))
    if name == "gaps":        # long runs of vertices without edges between the rows
        n = 3001
        u = np.arange(0, 2990, 230)
        return Graph(n, *edges_to_csr(n, u[:-1], u[1:]))
    return tiny_graph(701, 3333, seed=3)


@pytest.mark.parametrize("name", ["star", "gaps", "tiny"])
@pytest.mark.parametrize("S,k", [(1, 3), (1, 0), (2, 5), (3, 4), (16, 1)])
def test_every_split_gives_the_oracles_epoch(cuda, name, S, k):
    """Every number of edges per lane, one block and many: the same bits, and
    the oracle's positions within the parity gate."""
    g = _graph(name)
    Y0 = initial_positions(g.n, 5)
    sched = snap.linear_schedule(eta0=0.2, total_epochs=4)
    got = [gpu_layout(cuda, g, Y0, 1, k, sched, seed=6,
                      opts=snap.make_options(mode=snap.MODE_SYNC, sync_substeps=S, sync_cap=1.0, segment_edges=seg,
                                             block_threads=block))
           for seg, block in ((0, 0), (4, 32), (12, 0), (64, 96), (4096, 256))]
    for other in got[1:]:
        assert np.array_equal(got[0].view(np.uint32), other.view(np.uint32))
    ref = oracle.sync(g.row_ptr, g.col_idx, g.n, Y0, 1, k, schedule_dict(sched), seed=6, substeps=S, cap=1.0)
    assert parity_error(got[0], ref) < SYNC_RTOL
