"""Alg. 3 walks with trees and records in shared memory: both precisions,
classification and regression, trees of few splits and of the greatest depth,
trees and records too large for it, rows that end inside a segment of 2048 and
inside a group of 3; every importance row against the CPU oracle."""
import numpy as np
import pytest

from paper_2605_09950_gb300 import synth
from test_gpu_parity import built, check_iteration  # noqa: F401

pytestmark = pytest.mark.gpu


def workload(N, p, classes, bins, n_trees, depth, mtry, seed):
    """classes = 1: regression.  Noise labels (deep trees), a few columns with signal."""
    rng = np.random.default_rng(seed)
    X = np.zeros((p, synth.pad16(N)), np.uint8)
    X[:, :N] = rng.integers(0, bins, size=(p, N))
    if classes == 1:
        y = X[0, :N].astype(np.int64) * 2**16 + rng.integers(-2**21, 2**21, N)
    else:
        y = rng.integers(0, classes, size=N).astype(np.uint8)
        y[:classes] = np.arange(classes)
        X[: max(1, p // 64), :N] = np.clip(X[: max(1, p // 64), :N] // 2 + y * (bins // (2 * classes)), 0, bins - 1)
    task = (synth.REGRESSION if classes == 1 else synth.CLASSIFICATION) | synth.PERMUT
    return synth.Workload("t", X, y, N, p, task, classes, bins, n_trees, depth, 2, seed=seed, mtry=mtry)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("N,p,classes,bins,depth,mtry", [
    (8191, 12, 3, 64, 12, 5),      # just below the smallest of the shared-memory walks
    (8192, 12, 3, 2, 12, 1),       # few splits
    (8192, 12, 3, 64, 11, 5),      # the deepest trees that stay out
    (8201, 5, 2, 2, 30, 3),        # repeated features on every path, greatest depth
    (9003, 40, 5, 256, 20, 6),
    (9003, 40, 8, 64, 14, 40),
    (8500, 20, 1, 128, 16, 10),    # regression
    (8300, 1024, 2, 16, 13, 9),    # records of 2048 bytes, the longest staged
    (8300, 1030, 2, 16, 13, 9),    # longer
    (60_001, 1000, 8, 256, 30, 2),  # more split nodes than fit beside records of 2000 bytes
])
def test_walks(N, p, classes, bins, depth, mtry, precision):
    w = workload(N, p, classes, bins, 1 if N > 50_000 else 3, depth, mtry, seed=N + p)
    check_iteration(w, precision=precision)
