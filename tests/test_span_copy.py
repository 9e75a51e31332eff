"""Which tiles of a general-layout call are brought by bulk copies, on the host: no copy
of whole 16-byte granules may reach outside the operands."""
import ctypes
import random
import subprocess

import pytest

from paper_1304_7054_gb300 import build as libbuild

SRC = """
#include "kron_span_copy.h"
extern "C" void edges(uintptr_t x0, int64_t batch, int64_t P, int64_t ldxp, int64_t xspan, int es, int* r) {
    const kron::SpanEdges e = kron::span_edges(x0, batch, P, ldxp, xspan, es);
    r[0] = e.head; r[1] = e.tail; r[2] = e.copies;
}
"""


@pytest.fixture(scope="module")
def edges(tmp_path_factory):
    d = tmp_path_factory.mktemp("span")
    (d / "e.cpp").write_text(SRC)
    subprocess.run(["g++", "-shared", "-fPIC", "-I", libbuild.CSRC, str(d / "e.cpp"), "-o", str(d / "e.so")], check=True)
    f = ctypes.CDLL(str(d / "e.so")).edges
    f.argtypes = [ctypes.c_size_t] + [ctypes.c_int64] * 4 + [ctypes.c_int, ctypes.c_void_p]

    def run(*a):
        r = (ctypes.c_int * 3)()
        f(*a, r)
        return list(r)
    return run


@pytest.mark.parametrize("es", [2, 4])
def test_copies_stay_inside_the_operands(edges, es):
    rng = random.Random(es)
    copied = refused = 0
    for _ in range(20000):
        xspan, batch, P = rng.randint(1, 40), rng.randint(1, 30), rng.randint(1, 6)
        ldxp = rng.choice([0, 1, 3, xspan, xspan, xspan + rng.randint(0, 9)])
        x0 = 4096 + es * rng.randint(0, 8)
        x1 = x0 + es * ((batch - 1) * ldxp + xspan)
        head, tail, copies = edges(x0, batch, P, ldxp, xspan, es)
        ntiles = -(-batch // P)
        outside = []
        for t in range(ntiles):
            cnt = min(P, batch - t * P)
            b0 = x0 + es * t * P * ldxp
            b1 = b0 + es * ((cnt - 1) * ldxp + xspan)
            outside.append(b0 // 16 * 16 < x0 or -(-b1 // 16) * 16 > x1)
        assert head + tail <= ntiles and head <= 2 and tail <= 2
        assert copies == (0 if any(outside[head:ntiles - tail]) else 1)
        copied += copies * (ntiles - head - tail)
        refused += 1 - copies
        if xspan <= ldxp and (P * ldxp - (ldxp - xspan)) * es >= 16:   # operands one after the other
            assert copies
        if x0 % 16 == 0 and x1 % 16 == 0:
            assert (head, tail) == (0, 0)
    assert copied > 1000 and refused > 10
