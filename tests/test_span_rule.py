"""The rule that leaves calls of general layout to the scalar body, on the host: calls on
which both bodies were timed, on the side of the faster one."""
import ctypes
import subprocess

import pytest

from paper_1304_7054_gb300 import build as libbuild

SRC = """
#include "kron_span_rule.h"
extern "C" int scalar(int D, int es, int N, int64_t nx, int64_t ny, int64_t batch, int square, int up_one, int beta,
                      int x_packed, int y_packed, int y_aligned, int yvec, int row_bytes) {
    return kron::scalar_body_faster(kron::SpanCall{D, es, N, nx, ny, batch, square != 0, up_one != 0, beta != 0,
                                                   x_packed != 0, y_packed != 0, y_aligned != 0, yvec, row_bytes});
}
"""
LARGE = 1 << 25


@pytest.fixture(scope="module")
def scalar(tmp_path_factory):
    d = tmp_path_factory.mktemp("rule")
    (d / "r.cpp").write_text(SRC)
    subprocess.run(["g++", "-shared", "-fPIC", "-I", libbuild.CSRC, str(d / "r.cpp"), "-o", str(d / "r.so")], check=True)
    f = ctypes.CDLL(str(d / "r.so")).scalar
    f.argtypes = [ctypes.c_int] * 3 + [ctypes.c_int64] * 3 + [ctypes.c_int] * 8
    return f


def call(f, kind, es, x, y, batch=None, beta=0, x_packed=0, y_packed=0, y_aligned=0, yvec=0, ldy=None):
    nx, ny = x ** kind, y ** kind
    return bool(f(kind, es, max(x, y), nx, ny, batch or LARGE // max(nx, ny), x == y, y == x + 1, beta, x_packed,
                  y_packed, y_aligned, yvec, (ldy or y) * es))


# kind, bytes, n -> m, batch (None: large), beta, how Y lies; scalar / span time
MISALIGNED, PADDED, ROWS = {"x_packed": 1, "y_packed": 1}, {"x_packed": 1}, {}
SCALAR = [(2, 4, 7, 7, None, 1, MISALIGNED), (3, 4, 12, 12, None, 1, MISALIGNED), (3, 2, 13, 13, None, 1, MISALIGNED),
          (2, 2, 6, 6, None, 1, MISALIGNED), (2, 4, 5, 5, None, 1, PADDED), (3, 4, 9, 9, None, 1, PADDED),
          (2, 4, 16, 16, 100, 1, MISALIGNED), (3, 2, 10, 10, 100, 1, PADDED), (3, 4, 5, 5, None, 0, PADDED),
          (3, 2, 6, 6, None, 0, PADDED), (2, 4, 4, 4, 4, 0, ROWS), (3, 4, 3, 3, 16, 0, ROWS), (2, 2, 2, 2, 2000, 0, ROWS),
          (3, 2, 5, 9, 100, 0, ROWS), (3, 2, 3, 7, 2000, 0, ROWS), (3, 2, 6, 7, None, 1, ROWS), (2, 2, 5, 6, None, 1, ROWS),
          (3, 2, 13, 14, None, 1, ROWS), (3, 4, 6, 6, None, 1, ROWS), (3, 4, 1, 1, None, 0, ROWS),
          (3, 2, 6, 10, 100, 0, ROWS), (2, 2, 13, 11, 4, 0, ROWS), (2, 2, 9, 9, None, 1, MISALIGNED),
          (3, 2, 15, 15, None, 1, MISALIGNED), (2, 2, 14, 14, None, 1, {"x_packed": 1, "y_packed": 1, "yvec": 2})]
SPAN = [(2, 4, 16, 16, None, 1, MISALIGNED), (2, 2, 9, 9, None, 1, PADDED), (2, 4, 11, 11, None, 1, PADDED),
        (3, 4, 16, 16, None, 1, MISALIGNED), (2, 2, 12, 12, None, 1, PADDED),
        (2, 4, 7, 7, None, 0, MISALIGNED), (3, 2, 9, 9, None, 0, MISALIGNED), (2, 4, 12, 12, None, 0, PADDED),
        (2, 4, 7, 7, None, 1, ROWS), (3, 4, 8, 8, 100, 0, ROWS), (3, 4, 8, 12, 100, 0, ROWS), (2, 4, 4, 5, 2000, 0, ROWS),
        (3, 2, 12, 10, None, 1, ROWS), (3, 2, 13, 14, None, 0, ROWS), (2, 2, 14, 16, None, 0, ROWS),
        (2, 2, 14, 15, None, 1, ROWS), (2, 2, 14, 14, None, 1, MISALIGNED), (3, 2, 15, 15, None, 1, PADDED),
        (3, 2, 16, 14, None, 0, ROWS),
        (3, 2, 7, 7, 40, 0, {"x_packed": 1, "y_packed": 1, "y_aligned": 1}),
        (2, 2, 3, 3, 1, 0, {"x_packed": 1, "y_packed": 1, "y_aligned": 1})]


@pytest.mark.parametrize("kind,es,x,y,batch,beta,how", SCALAR)
def test_scalar_body(scalar, kind, es, x, y, batch, beta, how):
    assert call(scalar, kind, es, x, y, batch, beta, **how)


@pytest.mark.parametrize("kind,es,x,y,batch,beta,how", SPAN)
def test_span_body(scalar, kind, es, x, y, batch, beta, how):
    assert not call(scalar, kind, es, x, y, batch, beta, **how)
