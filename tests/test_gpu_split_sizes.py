"""Split kernels at the sizes where their layouts change: nodes of 8, 16, 32
and 64 rows (matrix-product split of few rows), samples around 32 features,
nodes of 128, 256, 1024 and 4096
rows (by-record split), 2 to 8 classes, coarse bins (exact ties) and fine ones; every tree against
the CPU oracle, bit for bit."""
import numpy as np
import pytest

from paper_2605_09950_gb300 import synth
from test_gpu_parity import built, check_iteration  # noqa: F401

pytestmark = pytest.mark.gpu


def workload(N, p, classes, bins, n_trees, depth, mtry, seed, importance=synth.TREEIMP):
    rng = np.random.default_rng(seed)
    y = rng.integers(0, classes, size=N).astype(np.uint8)
    y[:min(N, classes)] = np.arange(min(N, classes))
    X = np.zeros((p, synth.pad16(N)), np.uint8)
    X[:, :N] = rng.integers(0, bins, size=(p, N))
    X[: p // 3, :N] = np.clip(X[: p // 3, :N] // 2 + y * (bins // (2 * classes)), 0, bins - 1)
    return synth.Workload(f"N{N}", X, y, N, p, synth.CLASSIFICATION | importance, classes, bins, n_trees, depth, 2,
                          seed=seed, mtry=mtry)


@pytest.mark.parametrize("classes", [2, 3, 4, 5, 6, 8])
@pytest.mark.parametrize("N,bins,mtry", [(13, 3, 31), (26, 256, 33), (51, 7, 40), (66, 256, 5), (104, 16, 33),
                                         (410, 256, 32)])
def test_small_nodes(classes, N, bins, mtry):
    w = workload(N, 20, classes, bins, 24, 12, mtry, seed=N + classes)
    check_iteration(w, tie_break=classes & 1)


@pytest.mark.parametrize("classes", [2, 3, 5, 8])
@pytest.mark.parametrize("N,bins,mtry", [(205, 256, 33), (408, 60, 31), (415, 256, 7), (1650, 100, 40), (1622, 256, 3),
                                         (6480, 256, 5), (6700, 20, 34), (9000, 256, 4)])
def test_nodes_by_record(classes, N, bins, mtry):
    """In-bag roots around 128, 256, 1024 and 4096 rows (the tiles of the
    by-record kernels), more rows than the largest, bins of every lane width."""
    w = workload(N, 20, classes, bins, 5, 4, mtry, seed=N + classes)
    check_iteration(w, tie_break=classes & 1)


@pytest.mark.parametrize("tie_break", [0, 1])
@pytest.mark.parametrize("N,p,bins,discrete", [(13, 3, 3, 0), (30, 70, 2, 0), (900, 40, 3, 0), (900, 200, 3, 1),
                                               (2500, 130, 3, 0), (27_000, 5, 3, 0)])
def test_three_bin_regression(N, p, bins, discrete, tie_break):
    """Genotype columns: nodes of at most 8 rows, of one and several staged
    chunks and above the matrix-product kernel's largest (16384 rows); column
    counts around 128; few distinct targets (exact ties of unlike subsets)."""
    rng = np.random.default_rng(N + p)
    X = np.zeros((p, synth.pad16(N)), np.uint8)
    X[:, :N] = rng.integers(0, bins, size=(p, N))
    y = X[0, :N].astype(np.int64) * 3 - X[p // 2, :N] + (rng.integers(-2, 3, N) if discrete else 0)
    y = y * 2**20 + (0 if discrete else rng.integers(-2**23, 2**23, N))
    if N == 13:
        y = y * 2**33 - 2**55  # large targets: every limb in use
    w = synth.Workload("t", X, y.astype(np.int64), N, p, synth.REGRESSION | synth.TREEIMP, 1, bins, 6 if N < 5000 else 2,
                       9 if N < 5000 else 2, 2, seed=N, mtry=0)
    check_iteration(w, tie_break=tie_break)


@pytest.mark.parametrize("tie_break", [0, 1])
@pytest.mark.parametrize("N,p,bins,mtry,target", [(13, 20, 5, 0, "plain"), (51, 20, 256, 1 << 20, "plain"),
                                                  (60, 33, 40, 31, "wide"), (410, 12, 128, 1 << 20, "discrete"),
                                                  (415, 20, 7, 33, "plain"), (700, 20, 200, 0, "wide"),
                                                  (1650, 9, 256, 1 << 20, "plain"), (1700, 20, 100, 34, "discrete")])
def test_binned_regression(N, p, bins, mtry, target, tie_break):
    """Nodes around 8, 16, 32, 256 and 1024 rows; samples around 32 columns and
    all of them; targets of two and of three limbs, and few distinct ones."""
    rng = np.random.default_rng(N + p)
    X = np.zeros((p, synth.pad16(N)), np.uint8)
    X[:, :N] = rng.integers(0, bins, size=(p, N))
    y = X[0, :N].astype(np.int64) - 2 * X[p // 2, :N]
    if target == "discrete":
        y = rng.integers(-2, 3, N) * 2**20
    else:
        y = y * 2**16 + rng.integers(-2**21, 2**21, N)
    if target == "wide":
        y = y * 2**22 - 2**44
    w = synth.Workload("t", X, y.astype(np.int64), N, p, synth.REGRESSION | synth.TREEIMP, 1, bins, 6, 8, 2, seed=N,
                       mtry=mtry)
    check_iteration(w, tie_break=tie_break)


@pytest.mark.parametrize("classes", [2, 3, 5, 8])
@pytest.mark.parametrize("N,bins,mtry", [(4097, 256, 7), (5001, 33, 40), (66_000, 256, 3)])
def test_nodes_by_column(classes, N, bins, mtry):
    """Columns in shared memory: just above the largest tile, an odd number of
    rows, and roots whose weight exceeds the packed counts' 16 bits."""
    w = workload(N, 12, classes, bins, 3, 3, mtry, seed=N + classes)
    check_iteration(w, tie_break=classes & 1)
