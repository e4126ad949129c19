"""Regression over more than 4 bins, at the sizes where a node's kernel changes
with the rows and the sampled columns (reg_record_pays, reg_rows_pays): nodes of
33 to 1024 rows by blocks or by the column gathers, nodes of at most 32 rows by
matrix products or by row; genotype columns on both sides of three_bins_pay;
levels of many nodes, whose lists a kernel of their own writes; trees against the CPU oracle, bit for bit."""
import numpy as np
import pytest

from paper_2605_09950_gb300 import synth
from test_gpu_parity import built, check_iteration  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tie_break", [0, 1])
@pytest.mark.parametrize("N,mtry,bins,depth", [
    (1024, 1, 128, 9), (1025, 8, 128, 9), (1025, 9, 5, 9),  # blocks; gathers and products; blocks
    (2048, 10, 256, 10), (2049, 10, 64, 10), (2049, 17, 7, 10), (2944, 23, 256, 10),  # then by row
    (15_003, 30, 128, 8), (5003, 64, 33, 8)])
def test_regression_routes(N, mtry, bins, depth, tie_break):
    p = 40
    rng = np.random.default_rng(N + mtry)
    X = np.zeros((p, synth.pad16(N)), np.uint8)
    X[:, :N] = rng.integers(0, bins, size=(p, N))
    y = X[0, :N].astype(np.int64) * 2**17 - X[7, :N].astype(np.int64) * 2**16 + rng.integers(-2**21, 2**21, N)
    w = synth.Workload("t", X, y, N, p, synth.REGRESSION | synth.TREEIMP, 1, bins, 4, depth, 2, seed=N, mtry=mtry)
    check_iteration(w, tie_break=tie_break)


@pytest.mark.parametrize("tie_break", [0, 1])
@pytest.mark.parametrize("N,p,bins,n_trees,depth", [
    (2500, 20, 3, 40, 9), (2500, 20, 3, 41, 9), (17_001, 60, 3, 4, 6),  # records; by row (13 and 40 columns)
    (16_400, 150, 3, 2, 13), (27_000, 150, 2, 2, 13),  # records, and nodes of more than 16383 rows by column
    (16_400, 150, 3, 2, 5), (8200, 70, 3, 3, 2)])  # shallow: by row
def test_three_bin_routes(N, p, bins, n_trees, depth, tie_break):
    rng = np.random.default_rng(N + p)
    X = np.zeros((p, synth.pad16(N)), np.uint8)
    X[:, :N] = rng.integers(0, bins, size=(p, N))
    y = X[0, :N].astype(np.int64) * 2**20 - X[7, :N].astype(np.int64) * 2**19 + rng.integers(-2**21, 2**21, N)
    w = synth.Workload("t", X, y, N, p, synth.REGRESSION | synth.TREEIMP, 1, bins, n_trees, depth, 2, seed=N, mtry=0)
    check_iteration(w, trees=[0, n_trees - 1], tie_break=tie_break)


@pytest.mark.parametrize("N,mtry,n_trees,depth", [(700, 9, 130, 9), (3000, 12, 64, 10)])
def test_levels_of_many_nodes(N, mtry, n_trees, depth):
    p, bins = 30, 64
    rng = np.random.default_rng(N)
    X = np.zeros((p, synth.pad16(N)), np.uint8)
    X[:, :N] = rng.integers(0, bins, size=(p, N))
    y = X[0, :N].astype(np.int64) * 2**17 + rng.integers(-2**21, 2**21, N)
    w = synth.Workload("t", X, y, N, p, synth.REGRESSION | synth.TREEIMP, 1, bins, n_trees, depth, 2, seed=N, mtry=mtry)
    check_iteration(w, trees=[0, 1, n_trees - 1])
