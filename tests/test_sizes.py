"""The buffers of a session hold the augmented matrix of every iteration: the
library's bound on its columns, compiled as plain C++, against the oracle's
shadow counts over every number of live columns."""
import os
import subprocess

import pytest

import oracle

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_09950_gb300", "csrc")


@pytest.fixture(scope="module")
def sizes(tmp_path_factory):
    """{p: (shadow_count(p), max_augmented(p))} by the library's header."""
    d = tmp_path_factory.mktemp("sizes")
    (d / "sizes.cpp").write_text('#include <cstdio>\n#include "sizes.h"\nint main() { for (long p = 1; p <= 64; ++p) '
                                 'std::printf("%ld %ld %ld\\n", p, (long)bgb::shadow_count(p), (long)bgb::max_augmented(p)); }\n')
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(d / "sizes.cpp"), "-o", str(d / "sizes")], check=True)
    out = subprocess.run([str(d / "sizes")], check=True, capture_output=True, text=True).stdout
    return {int(a): (int(b), int(c)) for a, b, c in (line.split() for line in out.splitlines())}


def test_buffers_hold_every_live_count(sizes):
    for p, (shadows, most) in sizes.items():
        assert shadows == oracle.shadow_count(p)
        assert most == max(q + oracle.shadow_count(q) for q in range(1, p + 1)), p
    assert sizes[5][1] == 12 > 5 + sizes[5][0]  # one of five columns rejected: more columns than at first
    assert sizes[3][1] == 10 > 3 + sizes[3][0]
