"""Regression over two to four bins that samples less than an eighth of the
columns (the row-by-row kernel and the column gathers): every tree against the
CPU oracle, bit for bit, and the same again in a second iteration over the
memory of the first."""
import numpy as np
import pytest

from paper_2605_09950_gb300 import boruta, synth
from test_gpu_parity import built, check_iteration  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tie_break", [0, 1])
@pytest.mark.parametrize("bins", [2, 3, 4])
@pytest.mark.parametrize("N,mtry", [(13, 4), (60, 4), (700, 3), (3001, 4)])
def test_few_bins(N, mtry, bins, tie_break):
    p = 20
    rng = np.random.default_rng(N + bins)
    X = np.zeros((p, synth.pad16(N)), np.uint8)
    X[:, :N] = rng.integers(0, bins, size=(p, N))
    y = X[0, :N].astype(np.int64) * 2**20 + X[7, :N].astype(np.int64) * 2**19 + rng.integers(-2**21, 2**21, N)
    w = synth.Workload("t", X, y, N, p, synth.REGRESSION | synth.TREEIMP, 1, bins, 12, 11, 3, seed=N, mtry=mtry)
    S, P, state, imp = check_iteration(w, tie_break=tie_break)
    nodes = S.dump(boruta.DUMP_NODES, boruta.NODE_DTYPE)
    assert (nodes["bin"] < bins - 1).all()
    S.write(state)
    S.step()
    np.testing.assert_array_equal(S.dump(boruta.DUMP_NODES, boruta.NODE_DTYPE), nodes)
    np.testing.assert_array_equal(S.dump(boruta.DUMP_IMP, np.float64).reshape(imp.shape), imp)
