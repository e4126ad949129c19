"""The node dump holds exactly the nodes of the trees, for even and odd
numbers of trees (the node pool leaves places unused between levels)."""
import ctypes as ct

import numpy as np
import pytest

from paper_2605_09950_gb300 import boruta, synth
from test_gpu_parity import built, session  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("importance", [synth.TREEIMP, synth.PERMUT])
@pytest.mark.parametrize("n_trees", [1, 2, 3, 5, 8])
def test_node_dump_is_the_trees_nodes(n_trees, importance):
    w = synth.binary_small(N=200, p=8, n_inf=2, n_trees=n_trees, max_depth=5, max_iter=2, importance=importance)
    S = session(w)
    S.step()
    ptr = S.dump(boruta.DUMP_TREE_PTR, np.int64)
    levels = S.dump(boruta.DUMP_LEVELS, np.float64).reshape(-1, 3)
    nodes = S.dump(boruta.DUMP_NODES, boruta.NODE_DTYPE)
    assert len(nodes) == ptr[-1] == levels[:, 0].sum()
    assert (nodes["n_rows"] > 0).all()
    # a caller's buffer of the true size is taken and filled
    out = np.zeros(ptr[-1] + 1, boruta.NODE_DTYPE)
    out[-1]["n"] = 0xABCD
    need = ct.c_int64()
    rc = boruta.lib().boruta_session_dump(S._h, boruta.DUMP_NODES, out.ctypes.data, int(ptr[-1]) * out.itemsize,
                                          ct.byref(need))
    assert rc == 0 and need.value == int(ptr[-1]) * out.itemsize
    np.testing.assert_array_equal(out[:-1], nodes)
    assert out[-1]["n"] == 0xABCD
