"""Writes lockfree_small.npz: where the lock-free modes put the vertices of
small graphs, as the walks of commit 53d530d do (chunk by chunk, a small
graph's lanes in blocks of 256).

On several GB300s, with a build of that commit (GPUs differ by as much as two
runs on one do):
    PYTHONPATH=<checkout of 53d530d> python tests/golden/make_lockfree_small.py runs OUT.npz
then, anywhere:
    python tests/golden/make_lockfree_small.py merge OUT.npz ...

Per workload: the mean over all runs of the positions of the PINNED vertices
of highest degree (hubs are where the order of racing updates shows most), and
`own`, the median distance of two runs, on the same GPU or not.
"""
import os
import sys

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.append(os.path.join(HERE, ".."))

RUNS = 16


def runs(path):
    from lockfree_small import CASES, pinned, run_case
    np.savez(path, **{name: np.stack([run_case(name)[pinned(name)] for _ in range(RUNS)]).astype(np.float32)
                      for name in CASES})


def merge(paths):
    files = [np.load(p) for p in paths]
    out = {}
    for name in files[0].files:
        all_runs = np.concatenate([f[name] for f in files]).astype(np.float64)
        out[name] = all_runs.mean(axis=0).astype(np.float32)
        out[name + "_own"] = np.median([np.linalg.norm(all_runs[i] - all_runs[j])
                                        for i in range(len(all_runs)) for j in range(i)])
    np.savez_compressed(os.path.join(HERE, "lockfree_small.npz"), **out)


if __name__ == "__main__":
    runs(sys.argv[2]) if sys.argv[1] == "runs" else merge(sys.argv[2:])
