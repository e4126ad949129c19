"""Alg. 3 as printed where the device memory does not hold the table of leaf
values beside the forest: the session is accepted and gives the same run."""
import numpy as np
import pytest

from paper_2605_09950_gb300 import boruta, synth
from test_gpu_parity import built, session  # noqa: F401

pytestmark = pytest.mark.gpu


def test_printed_form_without_the_leaf_table():
    import torch

    C, trees, depth = 8, 200, 11
    w = synth.multiclass_toeplitz(N=2000, p=16, block=4, n_inf=3, n_classes=C, n_trees=trees, max_depth=depth, max_iter=2,
                                  importance=2)
    per_tree = sum(min(1 << level, w.N) for level in range(depth + 1))
    table = trees * per_tree * C * 8

    def run():
        S = session(w, permut_form=1, forest_rows=16)
        left = torch.cuda.mem_get_info()[0]
        S.step()
        out = S.dump(boruta.DUMP_IMP, np.float64), S.dump(boruta.DUMP_NODES, np.uint8)
        S.close()
        return left, out

    run()  # the context, the kernels' own memory
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    left, want = run()
    taken = free - left
    assert taken > table > 32 << 20
    keep = torch.empty(free - (taken - table // 2), dtype=torch.uint8, device="cuda")  # half a table too little
    _, got = run()
    del keep
    torch.cuda.empty_cache()
    for a, b in zip(got, want):
        np.testing.assert_array_equal(a, b)
