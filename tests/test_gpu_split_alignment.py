"""Split-precision calls that run on the CUDA cores: the route does not depend on where Y
starts, only on the size (with a line that lies lower off a 16-byte boundary)."""
import pytest
import torch

import paper_1304_7054_gb300 as kg
from paper_1304_7054_gb300 import inputs

pytestmark = pytest.mark.gpu

DT = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


@pytest.mark.parametrize("kind,n,io", [(2, 1, "f32"), (2, 4, "f32"), (2, 9, "f32"), (2, 14, "f32"), (3, 2, "f32"),
                                       (3, 7, "f32"), (3, 11, "f32"), (2, 3, "bf16"), (2, 9, "f16"), (2, 11, "bf16"),
                                       (3, 4, "f16"), (3, 11, "bf16")])
@pytest.mark.parametrize("off", [1, 2, 3])
@pytest.mark.parametrize("batch", [67, 5000])
def test_misaligned_results_are_the_fp32_result(kind, n, io, off, batch):
    if kind == 3 and n > 4:
        batch = min(batch, 700)
    b = inputs.make_batch(kind, n, batch, seed=170 + n)
    X = torch.from_numpy(b.X).to(DT[io]).cuda()
    ext = dict(zip(("ma", "na", "mb", "nb", "mc", "nc"), [n] * 2 * kind))
    f = kg.kron2_batched if kind == 2 else kg.kron3_batched
    out = {}
    for compute in ("native", "bf16x3"):
        Y = torch.full((X.numel() + off + 16,), 7.0, dtype=DT[io], device="cuda")
        f(*b.comps(), X, Y[off:], batch=batch, compute=compute, **ext)
        out[compute] = Y
    assert torch.equal(out["native"], out["bf16x3"])
