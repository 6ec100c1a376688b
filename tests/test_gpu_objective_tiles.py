"""The exact objective at the edges of its tiles and chunks."""
import numpy as np
import pytest

import oracle
import paper_2608_01907_gb300 as snap
from synth import initial_positions, tiny_graph

pytestmark = pytest.mark.gpu

# FP32 terms within 8 x 2^-24, summed in FP32 over at most 256 pairs or a
# chunk's entries, then in FP64
PAIRS_RTOL = (256 + 8) * 2.0 ** -24


@pytest.mark.parametrize("sampler", [snap.SAMPLER_UNIFORM, snap.SAMPLER_DEGREE])
@pytest.mark.parametrize("n", [2, 255, 256, 257, 1025, 2500, 13_999, 14_001, 15_361])
def test_pair_sum_at_the_tile_edges(cuda, n, sampler):
    torch = cuda
    g = tiny_graph(n, 3 * n, seed=n)
    Y = 3.0 * initial_positions(g.n, 8)
    sampling = oracle.Sampler.degree(g.row_ptr) if sampler == snap.SAMPLER_DEGREE else None
    ref = oracle.objective(g.row_ptr, g.col_idx, g.n, Y, 3, sampler=sampling)
    with snap.Layout(g.row_ptr, g.col_idx, opts=snap.make_options(sampler=sampler)) as L:
        attr, rep, total = L.objective(torch.from_numpy(Y).cuda(), 3)
    assert attr == pytest.approx(ref["attr"], rel=PAIRS_RTOL)
    assert rep == pytest.approx(ref["rep"], rel=PAIRS_RTOL)
    assert total == attr + rep


@pytest.mark.parametrize("keep", [False, True])
@pytest.mark.parametrize("n,m,seg", [(2, 0, 0), (40, 3, 4), (700, 2000, 0), (700, 2000, 12), (3000, 9001, 4096)])
def test_attraction_sum_over_short_chunks_and_groups(cuda, n, m, seg, keep):
    """Every edge once, whatever the chunks; the unused places of the last chunk are left out."""
    torch = cuda
    g = tiny_graph(n, m, seed=n + m)
    Y = 3.0 * initial_positions(g.n, 8)
    with snap.Layout(g.row_ptr, g.col_idx, opts=snap.make_options(segment_edges=seg, keep_csr=keep)) as L:
        attr, _, _ = L.objective(torch.from_numpy(Y).cuda(), 3)
    ref = oracle.objective(g.row_ptr, g.col_idx, g.n, Y, 3)["attr"]
    assert attr == pytest.approx(ref, rel=((seg or 4) + 16) * 2.0 ** -24)
