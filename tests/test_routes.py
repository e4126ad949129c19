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


# walks_pay(classification, fp32, N, trees, depth)
WALKS = [("walks_pay(true, true, 1000000, 300, 20)", 1), ("walks_pay(true, true, 100000, 500, 16)", 1),
         ("walks_pay(true, true, 100000, 100, 20)", 1), ("walks_pay(true, true, 20000, 100, 20)", 1),
         # few trees, few rows: one block after another
         ("walks_pay(true, true, 8192, 1, 20)", 0), ("walks_pay(true, true, 8192, 100, 16)", 0),
         ("walks_pay(true, true, 100000, 10, 16)", 0), ("walks_pay(true, true, 8191, 100000, 20)", 0),
         # trees of few levels
         ("walks_pay(true, true, 1000000, 300, 12)", 0),
         # FP64 losses of classes, at any size
         ("walks_pay(true, false, 1000000, 300, 20)", 0), ("walks_pay(true, false, 100000, 100, 16)", 0),
         # regression
         ("walks_pay(false, false, 100000, 100, 16)", 1), ("walks_pay(false, true, 20000, 100, 16)", 0),
         ("walks_pay(false, false, 10000, 100, 16)", 0)]


def test_walks(tmp_path):
    check(tmp_path, WALKS)
