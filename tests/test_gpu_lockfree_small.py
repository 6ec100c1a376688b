"""Lock-free epochs of small graphs put the vertices where they always did.

What racing lanes read depends on when they run, so a change of a walk's
timing alone can move hubs by more than chance does.  The pinned layouts are
means over 32 runs; a run differs from another by `own`, so a mean over 8
differs from such a mean by about own * sqrt((1/8 + 1/32) / 2) = 0.28 own by
chance.  Twice `own` leaves room for walks of another speed, and is half of
what a single run may differ by.
"""
import os

import numpy as np
import pytest

from lockfree_small import CASES, pinned, run_case

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "lockfree_small.npz")
RUNS = 8


@pytest.mark.parametrize("name", list(CASES))
def test_small_lockfree_layouts_land_where_pinned(cuda, name):
    want = np.load(GOLDEN)[name].astype(np.float64)
    at = pinned(name)
    runs = np.stack([run_case(name)[at] for _ in range(RUNS)])
    own = np.median([np.linalg.norm(runs[i] - runs[j]) for i in range(RUNS) for j in range(i)])
    off = np.linalg.norm(runs.mean(axis=0) - want)
    print(f"{name}: off {off:.3e}, own {own:.3e}, ratio {off / own:.2f}")
    assert off <= 2.0 * own
