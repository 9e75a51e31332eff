"""Which calls the general-layout body is asked for, on the host: a tile or depth set for
packed calls of odd n with 16-bit storage keeps them on the body it was set for."""
import ctypes
import subprocess

import pytest

from paper_1304_7054_gb300 import build as libbuild

SRC = """
#include "kron_span_rule.h"
extern "C" int asked(int y_aligned, int N, int half, int beta, int tile_set) {
    return kron::span_body_asked(y_aligned != 0, N, half != 0, beta != 0, tile_set != 0);
}
"""


@pytest.fixture(scope="module")
def asked(tmp_path_factory):
    d = tmp_path_factory.mktemp("asked")
    (d / "a.cpp").write_text(SRC)
    subprocess.run(["g++", "-shared", "-fPIC", "-I", libbuild.CSRC, str(d / "a.cpp"), "-o", str(d / "a.so")], check=True)
    return ctypes.CDLL(str(d / "a.so")).asked


def test_set_tiles_stay_with_the_scalar_body(asked):
    assert asked(1, 7, 1, 0, 0) == 1      # odd, 16-bit, packed, nothing set
    assert asked(1, 7, 1, 0, 1) == 0      # a tile or depth set
    assert asked(1, 7, 1, 1, 0) == 0      # beta != 0
    assert asked(1, 8, 1, 0, 0) == 0 and asked(1, 7, 0, 0, 0) == 0
    for tile_set in (0, 1):
        assert asked(0, 7, 1, 0, tile_set) == 1 and asked(0, 16, 0, 1, tile_set) == 1   # general layouts
