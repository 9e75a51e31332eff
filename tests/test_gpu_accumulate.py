"""beta != 0 in the bodies that bring the old results in by bulk copy (2-D n = 10, 14 and
odd n, 2-D and 3-D): ragged batches, batches smaller than a tile, ring depths."""
import numpy as np
import pytest
import torch

import paper_1304_7054_gb300 as kg
from helpers import arith_factor, storage_excess
from paper_1304_7054_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,n", [(2, 3), (2, 9), (2, 10), (2, 14), (2, 15), (3, 3), (3, 7), (3, 15)])
@pytest.mark.parametrize("batch", [1, 5, 83, 4001])
@pytest.mark.parametrize("depth", [0, 1, 3])
def test_old_results_enter_once(kind, n, batch, depth):
    if kind == 3 and n > 9:
        batch = min(batch, 641)
    b = inputs.make_batch(kind, n, batch, seed=n + batch)
    y0 = np.random.default_rng(n).standard_normal(b.X.size).astype(np.float32)
    X, Y = torch.from_numpy(b.X).cuda(), torch.from_numpy(y0).cuda()
    ext = dict(zip(("ma", "na", "mb", "nb", "mc", "nc"), [n] * 2 * kind))
    f = kg.kron2_batched if kind == 2 else kg.kron3_batched
    try:
        kg.set_tile_config(kind, n, "f32", "native", 0, depth)
        f(*b.comps(), X, Y, batch=batch, alpha=-0.5, beta=2.0, **ext)
    finally:
        kg.set_tile_config(kind, n, "f32", "native", 0, 0)
    m = [M.reshape(n, n, order="F").astype(np.float64) for M in b.comps()][::-1]     # mode 1 first
    x = b.X.astype(np.float64).reshape([batch] + [n] * kind)
    eq = "pml,il,jm->pji" if kind == 2 else "pqml,il,jm,kq->pkji"
    ref = -0.5 * np.einsum(eq, x, *m, optimize=True).ravel() + 2.0 * y0
    absref = 0.5 * np.einsum(eq, abs(x), *map(abs, m), optimize=True).ravel()
    assert storage_excess(Y.cpu().numpy(), ref, absref, "f32", arith_factor(kind, n), abs(2.0 * y0)) <= 1.0
