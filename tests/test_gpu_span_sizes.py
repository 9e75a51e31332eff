"""General layouts at batches large enough for the span body at every size (small calls go
to the scalar body), and, for the same shapes, a few instances on the scalar body."""
import pytest

from test_gpu_span import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", [2, 3])
@pytest.mark.parametrize("n", range(2, 9))
def test_small_rectangular_fp32(kind, n):
    for m in {max(1, n - 4), max(1, n - 1), n, n + 1, n + 4, 16}:
        for batch in (3, 66001 // max(n, m) ** kind + 1):
            run(kind, [n] * kind, [m] * kind, batch, "f32", gap=0 if m != n else 1)


@pytest.mark.parametrize("io", ["bf16", "f16"])
@pytest.mark.parametrize("kind,n,m", [(2, 2, 3), (2, 4, 3), (2, 5, 8), (3, 2, 3), (3, 5, 4), (3, 7, 9), (3, 9, 5), (3, 8, 4),
                                      (3, 10, 12), (3, 13, 15), (3, 16, 13), (2, 13, 16)])
def test_rectangular_16bit(io, kind, n, m):
    per = max(n, m) ** kind
    for batch, ab in ((3, (1.0, 0.0)), ((1 << 20) // per + 1, (1.0, 0.0)), ((1 << 20) // per + 1, (-0.5, 2.0))):
        run(kind, [n] * kind, [m] * kind, batch, io, alpha=ab[0], beta=ab[1])


@pytest.mark.parametrize("io", ["f32", "bf16"])
@pytest.mark.parametrize("kind,n", [(2, 3), (2, 12), (2, 16), (3, 7), (3, 12), (3, 16)])
@pytest.mark.parametrize("off", [1, 2, 8])
def test_packed_results_at_any_alignment(io, kind, n, off):
    """Packed operands and results whose base is off a 16-byte boundary (both bodies, by size)."""
    for batch in (5, 600_000 // n ** kind):
        for ab in ((1.0, 0.0), (-0.5, 2.0)):
            run(kind, [n] * kind, [n] * kind, batch, io, off=off, alpha=ab[0], beta=ab[1])
