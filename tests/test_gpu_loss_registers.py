"""The loss's fused column pass, whose forward outputs stay in registers as the
adjoint's inputs (GPU): every column length, the narrowest tiles, and 2048
points on both sides of eight 128 KiB tiles to an SM, against float64.

Three transforms, each adding about one float32 rounding (2^-24) per radix-2
level, and the two products with w bound the relative error of y.
"""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_15437_gb300 import build
    build.build()
    import paper_2506_15437_gb300 as g
    return g


def _shapes():
    for ny in (32, 64, 128, 256, 512, 1024):
        yield ny, 64, 3
        yield ny, 16, 611
    yield from ((512, 2, 5), (1024, 2, 5), (1024, 8, 1), (2048, 2, 3), (2048, 8, 2), (2048, 256, 37), (2048, 256, 41))


@pytest.mark.parametrize("ny,nx,b", list(_shapes()))
def test_column_half(g, ny, nx, b):
    gen = torch.Generator(device="cuda").manual_seed(ny + 3 * nx + b)
    x = torch.randn(b, ny, nx, dtype=torch.complex64, device="cuda", generator=gen)
    w = torch.rand(b, ny, nx, device="cuda", generator=gen)
    plan = g.Plan(nx, ny, b)
    assert plan.weighted_power_adjoint_parts() > 0
    loss, y = plan.weighted_power_adjoint(x, w)
    X = torch.fft.fft2(x.cdouble())
    ref = torch.fft.ifft(w * X, dim=-2, norm="forward")
    assert (torch.linalg.norm(y - ref) / torch.linalg.norm(ref)).item() < (math.log2(nx) + 2 * math.log2(ny) + 2) * 2.0**-24
    ref = (w * (X.real**2 + X.imag**2)).sum()
    assert abs(loss - ref) / ref < 1e-6
    z = x.clone()
    plan.weighted_power_adjoint(z, w, z)
    assert torch.equal(z, y) and plan.status() == 0
    plan.close()
