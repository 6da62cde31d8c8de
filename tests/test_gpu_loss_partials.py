"""The loss partials of the fused column pass (GPU): a thread's chain of float
sums is at most 16 long, however many terms it holds (four at a time from 32).

A unit impulse at every slice's origin has the transform 1 everywhere, exactly,
so a partial is the sum of the weights alone, in the order the kernel adds them.
The first row block's weights, each thread's first term, are 2^25 and the others
1: behind 2^25 (ulp 4) a lone 1 is lost, and a chain of 16 loses 15 of 2^25 (the
sums over threads are exact): relative error at most 15 / 2^25.  Chains of 32 and
64 lose 31 and 63.
"""
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


# elements per thread: 16, 32, 32 and, with eight tiles to an SM, 64; 2048 with fewer: 16
@pytest.mark.parametrize("ny,nx,b,e", [(256, 64, 2, 16), (512, 64, 2, 32), (1024, 64, 2, 32), (2048, 256, 41, 64),
                                       (2048, 64, 2, 16)])
def test_chains_of_sixteen(g, ny, nx, b, e):
    x = torch.zeros(b, ny, nx, dtype=torch.complex64, device="cuda")
    x[:, 0, 0] = 1
    w = torch.ones(b, ny, nx, device="cuda")
    w[:, : ny // e] = 2.0**25
    plan = g.Plan(nx, ny, b)
    assert plan.weighted_power_adjoint_parts() > 0
    loss, _ = plan.weighted_power_adjoint(x, w)
    assert torch.equal(plan.execute(x), torch.ones_like(x))
    exact = w.double().sum()
    assert 0 <= ((exact - loss) / exact).item() <= 15 / 2.0**25
    assert plan.status() == 0
    plan.close()
