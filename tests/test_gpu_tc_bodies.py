"""The split tensor bodies themselves, at every size: the built-in route sends small n to
the CUDA cores, so the body is set here (variant in 2-D, warps per instance in 3-D).
Bounds as derived in test_gpu_tc."""
import contextlib

import numpy as np
import pytest

import paper_1304_7054_gb300 as kg
from helpers import max_norm_err, oracle_ref, storage_check, storage_x
from paper_1304_7054_gb300 import inputs
from test_gpu_fiber import run_gpu
from test_gpu_tc import bound

pytestmark = pytest.mark.gpu


@contextlib.contextmanager
def body(kind, n, io, which):
    kw = {"variant": which} if kind == 2 else {"compute_warps": which}
    kg.set_kernel_config(kind, n, io, "bf16x3", **kw)
    try:
        yield
    finally:
        kg.set_kernel_config(kind, n, io, "bf16x3")


def check(Y, b, X64, io):
    if io == "f32":
        err = max_norm_err(Y, oracle_ref(b, X64), b, X64)
        assert err <= bound(b.kind, b.n)
        assert b.n < 2 or err <= 1e-5, err
    else:
        assert storage_check(Y, b, X64, io, compute="bf16x3") <= 1.0


CASES = [(2, "in_place"), (3, 1), (3, 4)]


@pytest.mark.parametrize("io", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("kind,which", CASES)
@pytest.mark.parametrize("n", range(1, 17))
def test_every_size(kind, which, n, io):
    b = inputs.make_batch(kind, n, 1037 if kind == 2 else 71, seed=700 + n, x_dist="normal")
    with body(kind, n, io, which):
        Y, X64 = run_gpu(b, io=io, compute="bf16x3", guard=16)
    check(Y, b, X64, io)


@pytest.mark.parametrize("io", ["f32", "bf16"])
@pytest.mark.parametrize("n", [3, 8, 10, 12])
@pytest.mark.parametrize("batch", [1, 3, 4099])
@pytest.mark.parametrize("warps", [1, 2, 8])
def test_3d_ragged_and_wrapping_batches(n, batch, warps, io):
    b = inputs.make_batch(3, n, batch, seed=720 + batch + n, x_dist="normal")
    with body(3, n, io, warps):
        Y, X64 = run_gpu(b, io=io, compute="bf16x3", guard=16)
    check(Y, b, X64, io)


@pytest.mark.parametrize("io", ["f32", "bf16"])
@pytest.mark.parametrize("kind,which", CASES)
@pytest.mark.parametrize("n", [1, 2, 4, 5, 7, 9, 10, 14])
def test_alpha_beta(kind, which, n, io):
    b = inputs.make_batch(kind, n, 99 if kind == 2 else 37, seed=740 + n, x_dist="normal")
    Y0 = np.random.default_rng(1).standard_normal(b.batch * n ** kind).astype(np.float32)
    if io != "f32":
        Y0 = storage_x(inputs.Batch(kind, n, b.batch, b.A, b.B, b.C, Y0), io)[1]
    Y0 = np.asarray(Y0, np.float64)
    with body(kind, n, io, which):
        Y, X64 = run_gpu(b, io=io, compute="bf16x3", alpha=0.75, beta=-2.0, Y0=Y0, guard=8)
    # element by element: the bound counts the rounding of beta Y0, which a bar normalised by
    # the components' norms does not (n = 1: their product is 1e-3 of beta Y0)
    assert storage_check(Y, b, X64, io, compute="bf16x3", alpha=0.75, beta=-2.0, Y0=Y0) <= 1.0


@pytest.mark.parametrize("io", ["bf16", "f16"])
@pytest.mark.parametrize("kind,which", CASES)
@pytest.mark.parametrize("n", [3, 4, 6, 8, 12])
def test_identity_is_exact(kind, which, n, io):
    b = inputs.make_batch(kind, n, 201, seed=760)
    eye = np.eye(n).ravel(order="F").astype(np.float32)
    b.A, b.B = eye, eye.copy()
    if kind == 3:
        b.C = eye.copy()
    with body(kind, n, io, which):
        Y, X64 = run_gpu(b, io=io, compute="bf16x3")
    assert np.array_equal(Y, X64)


@pytest.mark.parametrize("n", [1, 4, 8, 11])
@pytest.mark.parametrize("P,depth", [(3, 1), (7, 2), (33, 3)])
def test_2d_any_tile_16bit(n, P, depth):
    """Odd tiles leave the last group of instances on a tile's diagonal half filled."""
    b = inputs.make_batch(2, n, 1001, seed=780 + n + P, x_dist="normal")
    kg.set_kernel_config(2, n, "bf16", "bf16x3", variant="in_place", instances_per_tile=P, pipeline_depth=depth)
    try:
        Y, X64 = run_gpu(b, io="bf16", compute="bf16x3", guard=16)
    finally:
        kg.set_kernel_config(2, n, "bf16", "bf16x3")
    check(Y, b, X64, "bf16")
