"""The structure forms of the calls (kron2_batched_args, kron3_batched_args): the same
status as the argument-by-argument form for valid and invalid arguments (no GPU)."""
import ctypes

import numpy as np
import pytest

import paper_1304_7054_gb300 as kg
from paper_1304_7054_gb300 import build as libbuild

COMP = np.eye(16, dtype=np.float32).tobytes()
BASE2 = dict(s=0, batch=0, X=0x10000, Y=0x90000, ldxp=16, ldyp=16, ar=1.0, ai=0.0, br=0.0, bi=0.0, ma=4, na=4, mb=4,
             nb=4, lda=4, ldb=4, ldx=4, ldy=4, io=0, comp=0, ta=b"N", tb=b"T", tx=b"N")
BASE3 = dict(s=0, batch=0, X=0x10000, Y=0x90000, ldxp=64, ldyp=64, ar=1.0, ai=0.0, br=0.0, bi=0.0, ma=4, na=4, mb=4,
             nb=4, mc=4, nc=4, lda=4, ldb=4, ldc=4, ldx=4, ldx2=16, ldy=4, ldy2=16, io=0, comp=0, ta=b"N", tb=b"T",
             tc=b"C")


@pytest.fixture(scope="module")
def lib():
    libbuild.build()
    return kg.load_library()


@pytest.mark.parametrize("over", [{}, {"ma": 17}, {"nb": 0}, {"lda": 3}, {"ldx": 3}, {"ldyp": 15}, {"batch": -1},
                                  {"io": 9}, {"io": 1, "comp": 1}, {"ta": b"X"}, {"batch": 2, "X": 0},
                                  {"batch": 1, "Y": 0x10004}])
def test_same_status_2d(lib, over):
    a = {**BASE2, **over}
    one = ctypes.c_double(1.0)
    p = ctypes.addressof(one)
    full = lib.kron2_batched(a["s"], a["ta"], a["tb"], a["tx"], a["ma"], a["na"], a["mb"], a["nb"], a["batch"], p, COMP,
                             a["lda"], COMP, a["ldb"], a["X"], a["ldx"], a["ldxp"], p, a["Y"], a["ldy"], a["ldyp"],
                             a["io"], a["comp"])
    assert lib.kron2_batched_args(kg._ARGS2.pack(*a.values()), COMP, COMP) == full


@pytest.mark.parametrize("over", [{}, {"mc": 17}, {"na": 0}, {"ldc": 3}, {"ldx2": 15}, {"ldy2": 15}, {"ldyp": 63},
                                  {"comp": 7}, {"tc": b"X"}, {"batch": 1, "Y": 0x10008}])
def test_same_status_3d(lib, over):
    a = {**BASE3, **over}
    one = ctypes.c_double(1.0)
    p = ctypes.addressof(one)
    full = lib.kron3_batched(a["s"], a["ta"], a["tb"], a["tc"], a["ma"], a["na"], a["mb"], a["nb"], a["mc"], a["nc"],
                             a["batch"], p, COMP, a["lda"], COMP, a["ldb"], COMP, a["ldc"], a["X"], a["ldx"], a["ldx2"],
                             a["ldxp"], p, a["Y"], a["ldy"], a["ldy2"], a["ldyp"], a["io"], a["comp"])
    assert lib.kron3_batched_args(kg._ARGS3.pack(*a.values()), COMP, COMP, COMP) == full


def test_null_structure(lib):
    assert lib.kron2_batched_args(None, COMP, COMP) == 1
    assert lib.kron3_batched_args(None, COMP, COMP, COMP) == 1
