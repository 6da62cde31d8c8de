"""The mixed-radix kernel over pairs of transforms where its groups do not come
out even (GPU): batches large enough for it, whose last CTA holds one
transform, half a group (every lane b empty), one more, or all but one; and
column slices whose last group is narrower.  The row lengths put every radix in
every stage position (first, middle, last, only) where a schedule has it, in
both compiled classes; the column lengths have every radix in each class.
describe() says that the kernel over pairs runs and how many transforms a CTA
takes, so a change of the rules cannot leave these cases to another kernel.

Against float64, worst transform; bar: tests/helpers.py's mixed-radix bound.
"""
import pytest

from tests.helpers import tol_any

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BUTTERFLIES = 160_000  # twice these fill the GPU: the plan takes the kernel over pairs


@pytest.fixture(scope="module")
def g():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_15437_gb300 import build
    build.build()
    import paper_2506_15437_gb300 as g
    return g


def check(g, nx, ny, batch, axis, remainder):
    """Both directions, out of place and in place; `remainder` of W transforms in the last group."""
    gen = torch.Generator(device="cuda").manual_seed(nx + 3 * ny + batch)
    x = torch.randn(batch, ny, nx, dtype=torch.complex64, device="cuda", generator=gen)
    dims = [d for d, n in ((-2, ny), (-1, nx)) if n > 1]
    for inverse in (False, True):
        plan = g.Plan(nx, ny, batch, inverse=inverse)
        d = plan.describe()[axis]
        assert d["mixed"] == 1 and d["mixed_lanes"] == 2 and remainder(d["mixed_w"])
        y = plan.execute(x)
        X = x.cdouble()
        ref = torch.fft.ifftn(X, dim=dims, norm="forward") if inverse else torch.fft.fftn(X, dim=dims)
        err = torch.linalg.vector_norm(y - ref, dim=dims) / torch.linalg.vector_norm(ref, dim=dims)
        assert err.max().item() <= tol_any(nx, ny)
        z = x.clone()
        plan.execute(z, out=z)
        assert torch.equal(z, y) and plan.status() == 0
        plan.close()


ROWS = [3, 5, 6, 7, 9, 10, 11, 12, 13, 50, 52, 75, 96, 120, 126, 140, 154, 182, 242, 375, 896, 972, 1029, 1050, 1134,
        1536, 1936, 1944, 2016, 2025, 2366, 2420, 3675, 3718, 3750, 5120, 7000]


@pytest.mark.parametrize("n", ROWS)
def test_rows(g, n):
    plan = g.Plan(n, 1, 32 * BUTTERFLIES // n)
    W = plan.describe()["x"]["mixed_w"]
    plan.close()
    assert W % 2 == 0
    base = (32 * BUTTERFLIES // n // W + 1) * W
    for rem in sorted({1, W // 2, W // 2 + 1, W - 1} - {0, W}):
        check(g, n, 1, base + rem, "x", lambda w: w == W and (base + rem) % w == rem)


COLS = [20, 22, 27, 50, 75, 81, 100, 126, 154, 686, 896, 1029, 1134, 1584, 1600, 1728, 1815, 1944, 2016, 2366, 2420,
        2700, 2704, 3675, 3750, 4394, 5120, 7000]


@pytest.mark.parametrize("n", COLS)
def test_columns(g, n):
    nx = 1024
    batch = 32 * BUTTERFLIES // (n * nx) + 1
    plan = g.Plan(nx, n, batch)
    W = plan.describe()["y"]["mixed_w"]
    plan.close()
    assert W >= 4 and W % 2 == 0
    for rem in sorted({2, W // 2, W // 2 + 2, W - 2} - {0, W}):
        check(g, nx + rem, n, batch, "y", lambda w: w == W and (nx + rem) % w == rem)
