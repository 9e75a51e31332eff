"""Which mixed-size launches take their tiles over instead of walking them, on the host."""
import ctypes
import subprocess

import pytest

from paper_1304_7054_gb300 import build as libbuild

SRC = """
#include "kron_varlen_rule.h"
extern "C" int over(int units, int tiles, int resident) { return kron::tiles_taken_over(units, tiles, resident); }
"""


@pytest.fixture(scope="module")
def over(tmp_path_factory):
    d = tmp_path_factory.mktemp("rule")
    (d / "r.cpp").write_text(SRC)
    subprocess.run(["g++", "-shared", "-fPIC", "-I", libbuild.CSRC, str(d / "r.cpp"), "-o", str(d / "r.so")], check=True)
    return ctypes.CDLL(str(d / "r.so")).over


def units(kinds, lo, hi):
    return sum(k * n * n for k in kinds for n in range(lo, hi + 1))


def test_sides(over):
    assert over(units((2, 3), 4, 16), 30000, 608) == 1    # a large mix
    assert over(units((3,), 16, 16), 10000, 608) == 1
    assert over(units((2, 3), 2, 6), 30000, 608) == 0     # little code
    assert over(units((3,), 8, 12), 400, 608) == 0        # few tiles: at most two for a CTA
    assert over(units((2,), 4, 16), 1000, 608) == 0
    assert over(units((2,), 4, 16), 1217, 608) == 1
