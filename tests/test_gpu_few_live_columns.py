"""Iterations with fewer than five live columns, whose augmented matrix may
have more columns than the first iteration's (4 + 8 after 5 + 5): every tree
and importance row, the statistic, hits and decisions against the CPU oracle."""
import numpy as np
import pytest

from paper_2605_09950_gb300 import boruta, synth
from test_gpu_parity import REL64, built, check_iteration, close  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("task", [synth.CLASSIFICATION | synth.TREEIMP, synth.CLASSIFICATION | synth.PERMUT,
                                  synth.REGRESSION | synth.TREEIMP])
@pytest.mark.parametrize("p,rejected", [(2, 1), (3, 1), (3, 2), (5, 1), (5, 2), (5, 4), (6, 2)])
def test_few_live_columns(p, rejected, task):
    N, bins, trees = 300, 20, 7
    rng = np.random.default_rng(17 * p + rejected)
    X = np.zeros((p, synth.pad16(N)), np.uint8)
    X[:, :N] = rng.integers(0, bins, size=(p, N))
    noise = rng.integers(-4, 5, N)
    y = (X[p - 1, :N].astype(np.int64) + noise) * 2**20 if task & 1 else (X[p - 1, :N] + noise > bins // 2).astype(np.uint8)
    w = synth.Workload("t", X, y, N, p, task, 1 if task & 1 else 2, bins, trees, 5, 6, seed=p + rejected, mtry=0)
    state = dict(decision=np.zeros(p, np.int8), hits=np.arange(p, dtype=np.int32) % 3,
                 imp_history=np.full((6, p), np.nan), shadow_max=np.full(6, np.nan), iterations=2)
    state["decision"][:rejected] = -1
    S, P, _, _ = check_iteration(w, state=state, t=3)
    o = P.iteration(3, state["decision"], state["hits"])
    s = S.dump(boruta.DUMP_STAT, np.float64)
    if task & 2:
        close(s, o["s"], 1e3 * REL64)
    else:
        np.testing.assert_array_equal(s, o["s"])
    g = S.read()
    np.testing.assert_array_equal(g["hits"], o["hits"])
    np.testing.assert_array_equal(g["decision"], o["state"])
