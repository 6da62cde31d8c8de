"""The mixed-radix kernels over pairs of transforms where their groups do not
come out even, against the FP64 oracle: row batches around the group size (one
transform, an odd one, one past a whole group), column widths that are not a
multiple of the group (odd ones too, whose rows are not 16-byte aligned),
four-step rows with an odd n1, single-stage lengths, the longest length, in
both directions and in place.

Bar: tests/helpers.py's mixed-radix bound, 2e-7 * log2 n per axis.
"""
import numpy as np
import pytest

import oracle
import synth
from tests.helpers import ORACLE_THREADS, tol_any, worst_rel_l2

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


def check(g, x, ref, nx, ny, inverse):
    plan = g.Plan(nx, ny, x.shape[0], inverse=inverse)
    d = torch.from_numpy(x).cuda()
    got = plan.execute(d).cpu().numpy()
    assert worst_rel_l2(got, ref, nx * ny) <= tol_any(nx, ny)
    plan.execute(d, out=d)
    assert np.array_equal(d.cpu().numpy(), got)
    assert plan.status() == 0
    plan.close()


ROWS = [(3, 1), (15, 129), (100, 1), (100, 41), (300, 27), (1000, 3), (1000, 613), (1001, 5), (2187, 3), (3000, 305),
        (4095, 1), (7007, 3), (14336, 1), (14300, 3)]


@pytest.mark.parametrize("n,rows", ROWS, ids=[f"{a}x{b}" for a, b in ROWS])
@pytest.mark.parametrize("inverse", [False, True])
def test_row_groups(g, n, rows, inverse):
    x = synth.uniform_complex((rows, n), seed=n + rows)
    check(g, x, oracle.fft1d_any(x, dir=1 if inverse else -1, threads=ORACLE_THREADS), n, 1, inverse)


# (ny, nx): mixed-radix columns, nx odd, 2 mod 4, narrower than a group
COLS = [(6, 2), (6, 3), (100, 33), (100, 35), (360, 1025), (1000, 5), (1080, 2049), (2160, 18), (4095, 7), (7200, 3),
        (14336, 2)]


@pytest.mark.parametrize("ny,nx", COLS, ids=[f"{a}x{b}" for a, b in COLS])
@pytest.mark.parametrize("inverse", [False, True])
def test_column_groups(g, ny, nx, inverse):
    x = synth.uniform_complex((2, ny, nx), seed=ny + nx)
    check(g, x, oracle.fft2d_any(x, dir=1 if inverse else -1, threads=ORACLE_THREADS), nx, ny, inverse)


# odd n1 (243 * 243, 98415 = 3^9 5), n1 = 2 mod 4 (130 * 130, 130 * 150)
@pytest.mark.parametrize("n,batch", [(59049, 3), (98415, 2), (130 * 130, 2), (150 * 130, 3)])
@pytest.mark.parametrize("inverse", [False, True])
def test_fourstep_groups(g, n, batch, inverse):
    x = synth.uniform_complex((batch, n), seed=n % 9973)
    n1, n2 = g.Plan(n, 1, 1).describe()["x"]["mixed_fourstep"]
    assert n1 * n2 == n
    check(g, x, oracle.fft1d_any(x, dir=1 if inverse else -1, threads=ORACLE_THREADS), n, 1, inverse)
