"""The row kernel a plan chooses where something asks for 16 elements per thread
(GPU; describe() only, nothing is transformed)."""
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


def rows(g, nx, ny, batch):
    plan = g.Plan(nx, ny, batch)
    d = plan.describe()["rows"]
    plan.close()
    return d["kernel"].split("<")[0], d["e"]


@pytest.mark.parametrize("nx,ny,batch", [(4096, 1, 4096), (4096, 1, 512), (4096, 4096, 1)])
def test_the_landing_ring_is_honoured_at_every_size(g, monkeypatch, nx, ny, batch):
    assert rows(g, nx, ny, batch) == ("k_rows", 32 if nx * ny * batch >= 1 << 24 else 16)
    monkeypatch.setenv("GB300FFT_RING", "1")
    assert rows(g, nx, ny, batch) == ("k_rows_ring", 16)
