"""Columns, rows and four-step passes of 512 to 4096 points with 32 and 64 elements per thread (GPU).

Each length sits on both sides of the rules that choose them (enough tiles for
the SMs, enough points for the rows), with the narrowest and widest tiles,
against float64.  Each of the log2(n) radix-2 levels adds at most about one
float32 rounding (2^-24) to the relative error, so log2(n) 2^-24 bounds it.
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


def _check(g, nx, ny, batch):
    gen = torch.Generator(device="cuda").manual_seed(nx * 31 + ny * 7 + batch)
    x = torch.randn(batch, ny, nx, dtype=torch.complex64, device="cuda", generator=gen)
    dims = [d for d, n in ((-2, ny), (-1, nx)) if n > 1]
    bound = math.log2(nx * ny) * 2.0**-24
    for inverse in (False, True):
        ref = torch.fft.ifftn(x.cdouble(), dim=dims, norm="forward") if inverse else torch.fft.fftn(x.cdouble(), dim=dims)
        plan = g.Plan(nx, ny, batch, inverse=inverse)
        y = plan.execute(x)
        assert (torch.linalg.norm(y - ref) / torch.linalg.norm(ref)).item() < bound
        z = x.clone()
        plan.execute(z, out=z)
        assert torch.equal(z, y) and plan.status() == 0
        plan.close()


@pytest.mark.parametrize("ny", [512, 1024, 2048])
@pytest.mark.parametrize("nx,batch", [(4, 1), (8, 37), (16, 152), (64, 3), (512, 5)])
def test_columns(g, ny, nx, batch):
    _check(g, nx, ny, batch)


@pytest.mark.parametrize("ny,batch", [(128, 1), (128, 37), (256, 20)])
def test_short_columns_with_tiles_to_spare(g, ny, batch):
    _check(g, 1024, ny, batch)


@pytest.mark.parametrize("nx,points", [(512, 1 << 20), (1024, 1 << 20), (4096, 1 << 24)])
@pytest.mark.parametrize("below", [0, 1])
def test_rows(g, nx, points, below):
    _check(g, nx, 1, points // nx - below)


@pytest.mark.parametrize("log2n", range(14, 25))
@pytest.mark.parametrize("batch", [1, 3])
def test_four_step(g, log2n, batch):
    _check(g, 1 << log2n, 1, batch)
