"""General layouts whose operands start or end inside a 16-byte granule: the bits of the
same call on aligned operands (the phase changes who loads an element, not the sums)."""
import numpy as np
import pytest
import torch

import paper_1304_7054_gb300 as kg

pytestmark = pytest.mark.gpu

DT = {"f32": torch.float32, "bf16": torch.bfloat16}


@pytest.mark.parametrize("io", ["f32", "bf16"])
@pytest.mark.parametrize("na,nb,ma,mb", [(1, 2, 2, 1), (3, 1, 2, 3), (5, 3, 4, 5), (7, 9, 9, 7), (12, 11, 11, 12)])
@pytest.mark.parametrize("batch,ldxp", [(1, None), (2, None), (151, None), (4001, None), (37, 0), (37, 1)])
def test_operand_phase_does_not_change_bits(io, na, nb, ma, mb, batch, ldxp):
    rng = np.random.default_rng(na * 100 + batch)
    A, B = rng.uniform(-1, 1, (ma, na)), rng.uniform(-1, 1, (mb, nb))
    step = na * nb if ldxp is None else ldxp
    count = (batch - 1) * step + na * nb
    x = torch.from_numpy(rng.standard_normal(count).astype(np.float32)).to(DT[io]).cuda()
    out = []
    for off in range(0, 16 // x.element_size()):
        X = torch.full((off + count,), float("nan"), device="cuda", dtype=DT[io])[off:]
        X.copy_(x)
        Y = torch.full((batch * ma * mb,), float("nan"), device="cuda", dtype=DT[io])
        kg.kron2_batched(A, B, X, Y, ma=ma, na=na, mb=mb, nb=nb, batch=batch, ldxp=step)
        out.append(Y)
    assert not bool(torch.isnan(out[0]).any())
    assert all(torch.equal(o, out[0]) for o in out[1:])
    assert kg.device_status() == 0
