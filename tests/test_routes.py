"""The rules that choose a call's kernels (csrc/routes.h, compiled as plain
C++), at sizes where both sides were measured: a call goes to the faster one."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_09950_gb300", "csrc")


def evaluate(expressions, where):
    lines = "".join(f'  std::printf("%d\\n", static_cast<int>(bgb::{e}));\n' for e in expressions)
    (where / "routes.cpp").write_text('#include <cstdio>\n#include "routes.h"\nint main() {\n' + lines + "}\n")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(where / "routes.cpp"), "-o", str(where / "routes")], check=True)
    out = subprocess.run([str(where / "routes")], check=True, capture_output=True, text=True).stdout
    return [int(v) for v in out.split()]


def check(where, cases):
    got = evaluate([e for e, _ in cases], where)
    assert [(e, g) for (e, _), g in zip(cases, got)] == [(e, int(want)) for e, want in cases]


# walks_pay(classes (0: regression), fp32, N, trees, depth)
WALKS = [("walks_pay(5, true, 1000000, 300, 20)", 1), ("walks_pay(2, true, 100000, 500, 16)", 1),
         ("walks_pay(5, true, 100000, 100, 20)", 1), ("walks_pay(2, true, 20000, 100, 20)", 1),
         ("walks_pay(8, true, 90320, 224, 12)", 1), ("walks_pay(4, true, 166321, 160, 13)", 1),
         # few trees, few rows: one block after another
         ("walks_pay(5, true, 8192, 1, 20)", 0), ("walks_pay(8, true, 8192, 100, 16)", 0),
         ("walks_pay(8, true, 100000, 10, 16)", 0), ("walks_pay(5, true, 8191, 100000, 20)", 0),
         # trees of few levels
         ("walks_pay(2, true, 198838, 99, 12)", 0), ("walks_pay(5, true, 130989, 265, 11)", 0),
         ("walks_pay(2, true, 14753, 172, 14)", 0),
         # FP64 losses of classes, at any size
         ("walks_pay(5, false, 1000000, 300, 20)", 0), ("walks_pay(2, false, 100000, 100, 16)", 0),
         # regression
         ("walks_pay(0, false, 100000, 100, 16)", 1), ("walks_pay(0, true, 20000, 100, 16)", 0),
         ("walks_pay(0, false, 10000, 100, 16)", 0)]


def test_walks(tmp_path):
    check(tmp_path, WALKS)


# columns_pay(N, trees, mtry, depth, classes), records_pay(N, trees, mtry, depth, classes)
LARGE_CLASSIFICATION = [
    ("columns_pay(30011, 100, 20, 14, 5)", 1), ("columns_pay(65535, 1, 1, 4, 5)", 1), ("columns_pay(80000, 60, 31, 12, 5)", 1),
    ("columns_pay(85895, 74, 7, 18, 5)", 1), ("columns_pay(100000, 500, 44, 16, 5)", 1), ("columns_pay(100000, 200, 31, 12, 5)", 1),
    ("columns_pay(100000, 1, 4, 12, 5)", 1), ("columns_pay(156675, 302, 22, 18, 5)", 1),
    ("columns_pay(100000, 30, 31, 12, 5)", 0), ("columns_pay(100000, 100, 10, 12, 5)", 0), ("columns_pay(100000, 200, 4, 12, 5)", 0),
    ("columns_pay(130000, 60, 31, 12, 5)", 0), ("columns_pay(78669, 33, 39, 6, 5)", 0), ("columns_pay(124008, 110, 13, 7, 5)", 0),
    ("columns_pay(130000, 200, 44, 12, 5)", 1), ("columns_pay(99934, 46, 37, 11, 2)", 1),
    ("columns_pay(85282, 99, 42, 6, 5)", 1), ("columns_pay(142259, 89, 43, 6, 2)", 0),
    ("columns_pay(105741, 39, 14, 15, 6)", 0), ("records_pay(219170, 76, 23, 16, 5)", 1),
    ("records_pay(4000, 1, 1, 12, 2)", 1), ("records_pay(1000000, 300, 31, 20, 5)", 1),
    ("records_pay(200000, 100, 31, 12, 5)", 1), ("records_pay(200000, 10, 63, 12, 5)", 1),
    ("records_pay(215719, 197, 15, 16, 2)", 1), ("records_pay(214267, 266, 21, 18, 2)", 1),
    ("records_pay(200000, 100, 10, 12, 5)", 0), ("records_pay(400000, 300, 10, 20, 5)", 0),
    ("records_pay(1000000, 10, 14, 12, 2)", 0), ("records_pay(400000, 10, 20, 12, 5)", 0),
    ("records_pay(221890, 97, 42, 8, 8)", 0), ("records_pay(225026, 115, 20, 18, 6)", 0)]


def test_large_classification(tmp_path):
    check(tmp_path, LARGE_CLASSIFICATION)


# reg_record_pays(N, trees, mtry), reg_rows_pays(N, mtry)
REGRESSION = [("reg_record_pays(1000, 100, 1)", 1), ("reg_record_pays(2000, 100, 24)", 1),
              ("reg_record_pays(10000, 100, 100)", 1), ("reg_record_pays(100000, 10, 133)", 1),
              ("reg_record_pays(5000, 1, 33)", 1), ("reg_record_pays(5000, 10, 48)", 1),
              ("reg_record_pays(2000, 100, 10)", 0), ("reg_record_pays(5000, 100, 33)", 0),
              ("reg_record_pays(20000, 10, 33)", 0), ("reg_record_pays(20000, 100, 33)", 0),
              ("reg_record_pays(100000, 100, 33)", 0),
              ("reg_rows_pays(1000, 1)", 1), ("reg_rows_pays(2000, 4)", 1), ("reg_rows_pays(20000, 33)", 1),
              ("reg_rows_pays(100000, 133)", 1), ("reg_rows_pays(20000, 10)", 0), ("reg_rows_pays(5000, 4)", 0)]


def test_regression(tmp_path):
    check(tmp_path, REGRESSION)


# three_bins_pay(N, trees, mtry, columns, depth)
THREE_BINS = [("three_bins_pay(20000, 100, 3335, 10006, 10)", 1), ("three_bins_pay(1000, 100, 6, 48, 10)", 1),
              ("three_bins_pay(5000, 10, 6, 48, 10)", 1), ("three_bins_pay(5000, 100, 133, 400, 10)", 1),
              ("three_bins_pay(16000, 100, 100, 100, 10)", 1), ("three_bins_pay(40000, 100, 100, 400, 10)", 1),
              ("three_bins_pay(2000, 100, 16, 48, 10)", 1), ("three_bins_pay(2000, 300, 40, 120, 10)", 1),
              ("three_bins_pay(30000, 100, 66, 200, 10)", 1), ("three_bins_pay(2000, 300, 16, 48, 10)", 0),
              ("three_bins_pay(5000, 100, 24, 48, 10)", 0), ("three_bins_pay(16000, 100, 33, 100, 10)", 0),
              ("three_bins_pay(40000, 10, 33, 100, 10)", 0), ("three_bins_pay(40000, 1, 500, 4000, 10)", 0),
              ("three_bins_pay(300, 10, 10, 100, 10)", 0),
              ("three_bins_pay(20000, 100, 3335, 10006, 12)", 1), ("three_bins_pay(16000, 30, 133, 400, 6)", 1),
              ("three_bins_pay(8000, 3, 66, 200, 6)", 1), ("three_bins_pay(1000, 3, 66, 200, 2)", 1),
              ("three_bins_pay(8000, 100, 66, 200, 2)", 1), ("three_bins_pay(16000, 100, 133, 400, 4)", 1),
              ("three_bins_pay(70000, 30, 133, 400, 10)", 1), ("three_bins_pay(70709, 31, 100, 302, 4)", 0),
              ("three_bins_pay(103679, 14, 64, 194, 4)", 0), ("three_bins_pay(8000, 10, 400, 1200, 4)", 0),
              ("three_bins_pay(16000, 3, 400, 1200, 6)", 0), ("three_bins_pay(70000, 3, 66, 200, 8)", 0)]


def test_three_bins(tmp_path):
    check(tmp_path, THREE_BINS)


# lists_apart(regression, three_bins, reg_rows, nodes)
LISTS = [("lists_apart(true, false, true, 25600)", 1), ("lists_apart(true, false, true, 16384)", 0),
         ("lists_apart(true, false, false, 10)", 1), ("lists_apart(true, true, false, 25600)", 0),
         ("lists_apart(false, false, false, 25600)", 0)]


def test_lists(tmp_path):
    check(tmp_path, LISTS)
