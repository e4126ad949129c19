"""Alg. 3 walks with trees and records in shared memory, on forests large
enough for them (walks_pay): trees of few splits and of the greatest depth,
trees and records too large for it, rows that end inside a segment of 2048 and
inside a group of 3; importance rows of sampled trees against the CPU oracle."""
import pytest

from test_gpu_parity import built, check_iteration  # noqa: F401
from test_gpu_walks import workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,p,classes,bins,depth,mtry,rows,precision", [
    (8192, 12, 3, 2, 20, 1, 2_000_000, 1),      # few splits
    (8201, 5, 2, 2, 30, 3, 2_000_000, 1),       # repeated features on every path, greatest depth
    (9003, 40, 5, 256, 20, 6, 2_000_000, 1),
    (9003, 40, 8, 64, 20, 40, 2_000_000, 1),
    (8300, 1024, 2, 16, 20, 9, 2_000_000, 1),   # records of 2048 bytes, the longest staged
    (8300, 1030, 2, 16, 20, 9, 2_000_000, 1),   # longer
    (60_001, 1000, 8, 256, 30, 2, 2_000_000, 1),  # more split nodes than fit beside records of 2000 bytes
    (9003, 40, 5, 256, 16, 6, 3_000_000, 1),
    (9003, 40, 8, 256, 14, 6, 6_750_000, 1),
    (50_001, 20, 1, 128, 16, 10, 10_000_000, 0),  # regression
    (50_001, 20, 1, 128, 16, 10, 10_000_000, 1),
])
def test_walks(N, p, classes, bins, depth, mtry, rows, precision):
    n_trees = -(-rows // N)
    w = workload(N, p, classes, bins, n_trees, depth, mtry, seed=N + p)
    check_iteration(w, trees=[0] if N > 60_000 else [0, n_trees // 2, n_trees - 1], precision=precision)
