"""Classification of many rows that samples few columns: nodes of all sizes by
the column gathers alone (packed class weights below 4096, wide ones above),
and by record where the columns do not fit in shared memory; every tree against
the CPU oracle, bit for bit."""
import pytest

from test_gpu_parity import built, check_iteration  # noqa: F401
from test_gpu_split_sizes import workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("classes,N,p,bins,n_trees,depth,mtry", [
    (2, 90_001, 6, 256, 4, 9, 5), (3, 90_001, 6, 100, 4, 9, 3), (5, 81_920, 8, 256, 4, 10, 4), (8, 100_003, 6, 33, 4, 9, 5),
    (2, 210_001, 30, 256, 2, 10, 60),  # by record, columns longer than shared memory
    (5, 160_001, 30, 64, 2, 10, 60), (4, 200_001, 6, 256, 4, 10, 4),
    (2, 90_001, 6, 256, 30, 13, 12)])  # columns in shared memory beside the bands
def test_large_few_columns(classes, N, p, bins, n_trees, depth, mtry):
    w = workload(N, p, classes, bins, n_trees, depth, mtry, seed=N + classes)
    check_iteration(w, trees=[0, n_trees - 1], tie_break=classes & 1)
