"""The column-gather path (plan, histograms by feature band, exact argmax) on
the problems that still take it: regression that samples more than 512 columns
or has four bins, and classification on columns of at most four bins (two
classes counted in registers, three to five packed into 64-bit words, eight in
separate words).  In many chunks, by every launch form and every tuned tile
shape: trees and importances against the CPU oracle, and the same dumps."""
import numpy as np
import pytest

from paper_2605_09950_gb300 import boruta, synth
from test_gpu_parity import built, check_iteration, session  # noqa: F401

pytestmark = pytest.mark.gpu

CASES = {  # N, p, classes (1: regression), bins, mtry, smallest node of the path
    "regression, default sample of 533 of 1600 columns": (1200, 800, 1, 100, 0, 33),
    "regression, 513 of 600 columns": (700, 300, 1, 5, 513, 33),
    "regression, four bins": (1500, 40, 1, 4, 0, 33),
    "two classes, three bins": (3000, 40, 2, 3, 20, 65),
    "three classes, three bins": (3000, 40, 3, 3, 20, 65),
    "four classes, four bins": (2500, 30, 4, 4, 0, 65),
    "five classes, four bins, weight above the packed counts'": (7000, 20, 5, 4, 12, 65),
    "eight classes, two bins": (3000, 40, 8, 2, 20, 65),
}


@pytest.mark.parametrize("tie_break", [0, 1])
@pytest.mark.parametrize("case", CASES)
def test_band_path(case, tie_break):
    N, p, classes, bins, mtry, smallest = CASES[case]
    rng = np.random.default_rng(N + p + classes)
    X = np.zeros((p, synth.pad16(N)), np.uint8)
    X[:, :N] = rng.integers(0, bins, size=(p, N))
    if classes == 1:
        y = X[0, :N].astype(np.int64) * 2**17 - X[p // 2, :N].astype(np.int64) * 2**16 + rng.integers(-2**21, 2**21, N)
    else:
        y = ((X[0, :N] + 2 * X[1, :N] + rng.integers(0, classes, N)) % classes).astype(np.uint8)
    task = (synth.REGRESSION if classes == 1 else synth.CLASSIFICATION) | synth.TREEIMP
    w = synth.Workload("t", X, y, N, p, task, classes, bins, 3, 6, 2, seed=N, mtry=mtry)
    S, _, _, _ = check_iteration(w, tie_break=tie_break, chunk_nodes=3)
    nodes = S.dump(boruta.DUMP_NODES, boruta.NODE_DTYPE)
    taken = (nodes["n_rows"] >= smallest) & (nodes["feature"] >= 0)
    assert np.bincount(nodes["depth"][taken]).max() > 3 * 3  # a level in more than three chunks
    forms = {}
    for name, opts in dict(plain={}, per_band=dict(chunk_nodes=3, band_launch=1),
                           per_chunk=dict(chunk_nodes=3, band_launch=2), tuned=dict(autotune=1)).items():
        T = forms[name] = session(w, tie_break=tie_break, **opts)
        T.step()
        for what in (boruta.DUMP_NODES, boruta.DUMP_IMP, boruta.DUMP_STAT):
            np.testing.assert_array_equal(T.dump(what, np.uint8), S.dump(what, np.uint8), err_msg=name)
    # every chunk of a level is launched (a problem that other kernels take whole launches none)
    assert S.kernel_launches() > forms["plain"].kernel_launches() + 4 * 3
