"""Mixed-size plans whose resident CTAs walk the tile list in fixed steps, several tiles
each (few or small classes), and plans on either side of that rule, against the oracle."""
import numpy as np
import pytest
import torch


from helpers import torch_dtype
from test_gpu_varlen import bar, max_err, reference, run

pytestmark = pytest.mark.gpu


def mix(classes, count, seed):
    """`count` instances, every (kind, n) of `classes` equally often, in random order."""
    rng = np.random.default_rng(seed)
    comps = [[rng.uniform(-1, 1, n * n).astype(np.float32) for _ in range(k)] for k, n in classes]
    cls = rng.integers(0, len(classes), count).astype(np.int32)
    sizes = np.array([n ** k for k, n in classes], np.int64)[cls]
    off = np.concatenate([[0], np.cumsum(sizes)])
    X = rng.standard_normal(int(off[-1])).astype(np.float32)

    class V:
        pass
    v = V()
    v.classes, v.comps, v.class_of = classes, comps, cls
    v.x_off = v.y_off = off[:-1]
    v.X, v.total = X, int(off[-1])
    return v


PLANS = {"2d-6": ([(2, 6)], 100_000), "3d-8": ([(3, 8)], 20_000), "2d-2-4": ([(2, n) for n in (2, 3, 4)], 400_000),
         "mixed-2-4": ([(k, n) for k in (2, 3) for n in (2, 3, 4)], 200_000), "3d-5": ([(3, 5)], 60_000),
         "few-tiles": ([(k, n) for k in (2, 3) for n in range(8, 17)], 1500),
         "two-rounds": ([(2, n) for n in range(4, 17)], 20_000)}


@pytest.mark.parametrize("io", ["f32", "bf16"])
@pytest.mark.parametrize("name", PLANS)
def test_walked_plans(name, io):
    v = mix(*PLANS[name], seed=len(name))
    plan, X, Y, ws, X64 = run(v, io)
    idx = np.sort(np.random.default_rng(3).choice(len(v.class_of), min(len(v.class_of), 20000), replace=False))
    idx[-1] = len(v.class_of) - 1
    Yh = Y.double().cpu().numpy()
    assert not np.isnan(Yh).any()
    assert max_err(v, Yh, reference(v, X64, idx), io) <= bar(io)
    plan.close()


@pytest.mark.parametrize("io", ["f32", "bf16"])
def test_walked_plan_with_old_results(io):
    """alpha, beta over several tiles per CTA: beta Y enters once, on every instance (the plan's
    own plain results, rounded to the storage type, are the K x that is scaled)."""
    v = mix([(2, 6), (3, 4)], 150_000, seed=9)
    plan, X, Y, ws, _ = run(v, io)
    y0 = torch.randn(v.total, generator=torch.Generator().manual_seed(4)).to(torch_dtype(io)).cuda()
    Z = y0.clone()
    plan.set_scaling(-0.5, 2.0)
    plan.execute(X, Z, ws)
    # alpha and beta are powers of two: -0.5 K x and 2 y0 are exact, one FP32 sum, one rounding
    want = (-0.5 * Y.float() + 2.0 * y0.float()).to(torch_dtype(io))
    assert torch.equal(Z, want)
    plan.close()
