"""Writes lockfree_small.npz: where the lock-free modes put the vertices of
small graphs, as the walks of commit 53d530d do (one block of lanes after
another, chunk by chunk).

Run on a GB300 with a build of that commit:
    PYTHONPATH=<checkout of 53d530d> python tests/golden/make_lockfree_small.py
Each entry is the mean over RUNS runs of the positions of the PINNED vertices
of highest degree (hubs are where the order of racing updates shows most).
"""
import os
import sys

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.append(os.path.join(HERE, ".."))

RUNS = 32


def main():
    from lockfree_small import CASES, pinned, run_case
    out = {}
    for name in CASES:
        runs = np.stack([run_case(name) for _ in range(RUNS)])
        out[name] = runs[:, pinned(name)].mean(axis=0).astype(np.float32)
    np.savez_compressed(os.path.join(HERE, "lockfree_small.npz"), **out)


if __name__ == "__main__":
    main()
