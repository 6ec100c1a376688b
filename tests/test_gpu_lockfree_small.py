"""Lock-free epochs of small graphs put the vertices where they always did.

What racing lanes read depends on when they run, so a change of a walk's
timing alone can move hubs by more than chance does.  The pinned layouts are
means of former runs on three GPUs, and `own` is what two of those runs differ
by.  On each of those GPUs the former walk's own mean lies up to 1.1 `own` from
the mean of another; twice `own` leaves room for that and for walks of another
speed, and is half of what a single run may differ by.
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
    golden = np.load(GOLDEN)
    want, own = golden[name].astype(np.float64), float(golden[name + "_own"])
    at = pinned(name)
    off = np.linalg.norm(np.mean([run_case(name)[at] for _ in range(RUNS)], axis=0) - want)
    print(f"{name}: off {off:.3e}, own {own:.3e}, ratio {off / own:.2f}")
    assert off <= 2.0 * own
