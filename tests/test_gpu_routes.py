"""Calls that a rule sends to another kernel body: the split path's small sizes and the
balanced tiles of the FP64 bodies."""
import numpy as np
import pytest
import torch

import oracle
import paper_1304_7054_gb300 as kg
from paper_1304_7054_gb300 import inputs

pytestmark = pytest.mark.gpu

DT = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16, "f64": torch.float64}


def call(kind, n, batch, comps, X, Y, **kw):
    if kind == 2:
        return kg.kron2_batched(*comps, X, Y, ma=n, na=n, mb=n, nb=n, batch=batch, **kw)
    return kg.kron3_batched(*comps, X, Y, ma=n, na=n, mb=n, nb=n, mc=n, nc=n, batch=batch, **kw)


@pytest.mark.parametrize("kind,n,io", [(2, 1, "f32"), (2, 8, "f32"), (2, 15, "f32"), (3, 4, "f32"), (3, 14, "f32"),
                                       (2, 9, "bf16"), (2, 11, "f16"), (3, 5, "bf16"), (3, 12, "f16")])
def test_small_split_calls_are_the_fp32_result(kind, n, io):
    b = inputs.make_batch(kind, n, 67, seed=70 + n)
    X = torch.from_numpy(b.X).to(DT[io]).cuda()
    a, s = torch.empty_like(X), torch.empty_like(X)
    call(kind, n, 67, b.comps(), X, a)
    call(kind, n, 67, b.comps(), X, s, compute="bf16x3")
    assert torch.equal(a, s)


@pytest.mark.parametrize("kind", [2, 3])
def test_split_path_still_refuses_gaps(kind):
    b = inputs.make_batch(kind, 4, 5, seed=3)
    X = torch.zeros(5 * 4 ** kind + 64, device="cuda")
    with pytest.raises(kg.KronError) as e:
        call(kind, 4, 5, b.comps(), X, torch.zeros_like(X), compute="bf16x3", ldxp=4 ** kind + 4)
    assert e.value.status == 2


@pytest.mark.parametrize("kind", [2, 3])
@pytest.mark.parametrize("n", [1, 2, 3, 7, 9, 10, 12, 14, 15])
@pytest.mark.parametrize("batch", [1, 153, 2003])
def test_fp64_tiles(kind, n, batch):
    if kind == 3 and n > 9 and batch > 1000:
        batch = 700
    b = inputs.make_batch(kind, n, batch, seed=90 + n, dtype=np.float64)
    X = torch.from_numpy(b.X).cuda()
    Y = torch.full_like(X, float("nan"))
    call(kind, n, batch, b.comps(), X, Y)
    f = oracle.kron2 if kind == 2 else oracle.kron3
    ext = dict(zip(("ma", "na", "mb", "nb", "mc", "nc")[:2 * kind], [n] * 2 * kind))
    ref = f(*b.comps(), b.X, batch=batch, **ext)
    absref = f(*map(abs, b.comps()), abs(b.X), batch=batch, **ext)
    bound = 2 * kind * (n + 1) * 2.0 ** -53 * absref      # both sides: kind dot products of length n
    assert bool((np.abs(Y.cpu().numpy() - ref) <= bound).all())
