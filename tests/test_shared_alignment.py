"""Histograms in shared memory are read and written 16 bytes at a time
(`ld_bins`, `st_bins` and the helpers over them): an array that is declared on
its own, rather than in 16-byte aligned dynamic shared memory, must say so."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_09950_gb300", "csrc")
WIDE = r"(?:ld_bins|st_bins|record_prefix|record_best|record_zero)\s*(?:<[^<>;]*>)?\s*\(\s*(\w+)"


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu"))), ids=os.path.basename)
def test_static_histograms_are_aligned(path):
    text = re.sub(r"//[^\n]*", "", open(path).read())
    wide = set(re.findall(WIDE, text))
    for decl in re.findall(r"^\s*__shared__\s+([^;]*);", text, flags=re.M):
        arrays = set(re.findall(r"(\w+)\s*\[", decl))
        assert "__align__(16)" in decl or not (arrays & wide), decl


def test_the_check_sees_the_histograms():
    text = open(os.path.join(CSRC, "column.cu")).read()
    assert "hist" in re.findall(WIDE, text)
