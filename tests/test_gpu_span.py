"""General layouts on the GPU: rectangular components, gaps, transposed operands, any
alignment, ragged batches and 16-bit storage, element by element against a float64
einsum (the componentwise FP32 bound of helpers.storage_excess), gaps untouched."""
import numpy as np
import pytest
import torch

import paper_1304_7054_gb300 as kg
from helpers import arith_factor, storage_excess

pytestmark = pytest.mark.gpu

DT = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
FILL = 7.0


def run(kind, xe, ye, batch, io, tx=False, pad=0, gap=0, off=0, alpha=1.0, beta=0.0, variant=None):
    """xe, ye: extents per mode of op(X) and Y (mode 1 first)."""
    g = torch.Generator().manual_seed(kind * 1000 + 16 * xe[0] + ye[0])
    ms = [torch.rand(o, i, generator=g, dtype=torch.float32) * 2 - 1 for o, i in zip(ye, xe)]
    xs = [xe[1], xe[0]] if tx else list(xe)          # stored extents of X
    ldx, ldy = xs[0] + pad, ye[0] + pad
    ldxp, ldyp = ldx * int(np.prod(xs[1:])) + gap, ldy * int(np.prod(ye[1:])) + gap
    X = torch.randn(off + batch * ldxp, generator=g).to(DT[io])
    Y = torch.full((off + batch * ldyp,), FILL).to(DT[io])
    xv = X[off:].as_strided([batch] + xs[::-1], [ldxp] + ([ldx * xs[1]] if kind == 3 else []) + [ldx, 1]).double().numpy()
    shape, stride = [batch] + list(ye)[::-1], [ldyp] + ([ldy * ye[1]] if kind == 3 else []) + [ldy, 1]
    y0 = Y[off:].as_strided(shape, stride).double().numpy()
    if tx:
        xv = xv.transpose(0, 2, 1)
    m = [M.double().numpy() for M in ms]
    eq = "pml,il,jm->pji" if kind == 2 else "pqml,il,jm,kq->pkji"
    ref = alpha * np.einsum(eq, xv, *m, optimize=True) + beta * y0
    absref = abs(alpha) * np.einsum(eq, abs(xv), *map(abs, m), optimize=True)
    Xd, Yd = X.cuda(), Y.cuda()
    kw = dict(batch=batch, alpha=alpha, beta=beta, ldx=ldx, ldxp=ldxp, ldy=ldy, ldyp=ldyp)
    if kind == 2:
        kg.kron2_batched(ms[1], ms[0], Xd[off:], Yd[off:], ma=ye[1], na=xe[1], mb=ye[0], nb=xe[0],
                         transx="T" if tx else "N", **kw)
    else:
        kg.kron3_batched(ms[2], ms[1], ms[0], Xd[off:], Yd[off:], ma=ye[2], na=xe[2], mb=ye[1], nb=xe[1], mc=ye[0],
                         nc=xe[0], ldx2=ldx * xe[1], ldy2=ldy * ye[1], **kw)
    got = Yd.cpu()
    out = got[off:].as_strided(shape, stride)
    n = max(*xe, *ye)
    assert storage_excess(out.double().numpy(), ref, absref, io, arith_factor(kind, n),
                          abs(beta * y0) if (alpha, beta) != (1.0, 0.0) else None) <= 1.0
    mask = torch.zeros_like(got, dtype=torch.bool)
    mask[off:].as_strided(shape, stride)[...] = True
    assert bool((got[~mask] == FILL).all())           # nothing outside the results is written
    assert torch.equal(Xd.cpu(), X)


# every mode n -> m with |n - m| <= 4 has its own instantiation; beyond that, and for
# extents that differ per mode, the runtime-extent one runs
@pytest.mark.parametrize("kind", [2, 3])
@pytest.mark.parametrize("n", range(1, 17))
def test_rectangular(kind, n):
    for m in {1, max(1, n - 4), max(1, n - 1), n, min(16, n + 1), min(16, n + 4), 16}:
        run(kind, [n] * kind, [m] * kind, 5 if kind == 3 else 37, "f32", gap=0 if m != n else 1)


@pytest.mark.parametrize("io", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("kind,xe,ye", [(2, [16, 1], [1, 16]), (2, [3, 11], [14, 5]), (3, [1, 16, 2], [9, 1, 4]),
                                        (3, [5, 8, 13], [16, 2, 7]), (3, [16, 15, 14], [13, 16, 16])])
@pytest.mark.parametrize("pad,gap,off,ab", [(0, 0, 0, (1.0, 0.0)), (3, 5, 1, (1.0, 0.0)), (4, 8, 4, (-0.5, 2.0)),
                                            (0, 0, 3, (0.5, 0.0))])
def test_mixed_extents(io, kind, xe, ye, pad, gap, off, ab):
    for batch in (1, 3, 66):
        run(kind, xe, ye, batch, io, pad=pad, gap=gap, off=off, alpha=ab[0], beta=ab[1])


@pytest.mark.parametrize("io", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("n", [1, 2, 5, 8, 12, 15, 16])
@pytest.mark.parametrize("pad", [0, 1, 4])
def test_transposed_operand(io, n, pad):
    for off, batch, ab in ((0, 257, (1.0, 0.0)), (1, 40, (1.0, 0.0)), (0, 19, (2.0, -1.0))):
        run(2, [n, n], [n, n], batch, io, tx=True, pad=pad, off=off, alpha=ab[0], beta=ab[1])
    run(2, [n, min(16, n + 3)], [min(16, n + 1), n], 21, io, tx=True, pad=pad)


@pytest.mark.parametrize("io", ["bf16", "f16"])
@pytest.mark.parametrize("kind", [2, 3])
@pytest.mark.parametrize("n", [1, 3, 7, 9, 13, 15])
def test_odd_16bit_contiguous(io, kind, n):
    for batch in (1, 9, 515 if kind == 2 else 41):
        run(kind, [n] * kind, [n] * kind, batch, io)
        run(kind, [n] * kind, [n] * kind, batch, io, alpha=0.75, beta=1.5)


def test_non_finite_operands_stay_in_their_fibers():
    """An infinity reaches exactly the results that use it (no zero-padding product)."""
    X = torch.ones(8, 5, 3, device="cuda")
    X[2, 1, 1] = float("inf")
    Y = torch.zeros(8, 6, 4, device="cuda")
    A, B = np.ones((6, 5), np.float32), np.ones((4, 3), np.float32)
    kg.kron2_batched(A, B, X, Y, ma=6, na=5, mb=4, nb=3, batch=8)
    assert bool(torch.isinf(Y[2]).all()) and bool(torch.isfinite(Y[[0, 1, 3, 4, 5, 6, 7]]).all())
