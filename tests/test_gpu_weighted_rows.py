"""The adjoint under a weight array of plans whose 4096-point rows hold 32
elements per thread (GPU): the weighted pass keeps 16, the unweighted and the
scaled one do not, and each is right beside the others on one plan.

Bound: the gradient's 2 * 2e-7 * log2 N for two transforms, relative L2 against float64.
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


def rel(y, ref):
    return (torch.linalg.norm(y - ref) / torch.linalg.norm(ref)).item()


@pytest.mark.parametrize("nx,ny,b,e,we", [(4096, 4096, 1, 32, 16), (4096, 2048, 2, 32, 16), (4096, 2048, 1, 16, 16),
                                          (1024, 1024, 16, 32, 32), (512, 2048, 16, 32, 32), (4096, 8, 512, 32, 16)])
def test_weighted_adjoint(g, nx, ny, b, e, we):
    gen = torch.Generator(device="cuda").manual_seed(nx + ny + b)
    x = torch.randn(b, ny, nx, dtype=torch.complex64, device="cuda", generator=gen)
    w = torch.rand(b, ny, nx, device="cuda", generator=gen)
    scale = torch.tensor([0.75], device="cuda")
    plan = g.Plan(nx, ny, b)
    d = plan.describe()["rows"]
    assert (d["e"], d["weighted_e"]) == (e, we)
    bound = 2 * 2e-7 * math.log2(nx * ny)
    adjoint = torch.fft.ifft2(w * x.cdouble(), norm="forward")
    y = plan.execute(x)
    assert rel(plan.backward_weighted(x, w, 2.0), 2.0 * adjoint) <= bound
    assert rel(plan.backward_weighted_dev(x, w, scale, 2.0), 1.5 * adjoint) <= bound
    z = x.clone()
    assert torch.equal(plan.backward_weighted(z, w, 2.0, out=z), plan.backward_weighted(x, w, 2.0))
    assert torch.equal(plan.execute(x), y) and rel(y, torch.fft.fft2(x.cdouble())) <= bound
    if plan.weighted_power_adjoint_parts():
        rows = torch.fft.ifft(x.cdouble(), norm="forward")
        assert rel(plan.backward_rows_scaled(x, scale, 2.0), 1.5 * rows) <= bound
    assert plan.status() == 0
    plan.close()
