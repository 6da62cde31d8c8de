"""The one-pass Bluestein kernel over half-length transforms (padded length
M = 2Q, Q = 64 ... 8192) against the FP64 oracle, at the shortest and longest
lengths each Q takes, with a last CTA that is partly filled, both directions
and in place.

Bar: tests/helpers.py's Bluestein bound, 2e-7 * (3 log2 M + 3); the half-length
form runs one radix-2 level fewer at either end and adds two unit-modulus
factors, which the bound's three roundings and three full transforms cover.
"""
import numpy as np
import pytest

import oracle
import synth
from tests.helpers import ORACLE_THREADS, bluestein_m, tol_any, worst_rel_l2

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


LENGTHS = [n for q in (64, 128, 256, 512, 1024, 2048, 4096, 8192) for n in (q // 2 + 1, q - 1)]


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("inverse", [False, True])
def test_half_length_bluestein(g, monkeypatch, n, inverse):
    rows = 37 if n < 512 else 3
    x = synth.uniform_complex((rows, n), seed=50 + n)
    monkeypatch.setenv("GB300FFT_MIXED", "0")  # smooth lengths too
    plan = g.Plan(n, 1, rows, inverse=inverse)
    monkeypatch.delenv("GB300FFT_MIXED")
    d = plan.describe()["x"]
    assert d["bluestein_m"] == bluestein_m(n) and d["half_q"] == bluestein_m(n) // 2
    xd = torch.from_numpy(x).cuda()
    got = plan.execute(xd).cpu().numpy()
    ref = oracle.fft1d_any(x, dir=1 if inverse else -1, threads=ORACLE_THREADS)
    assert worst_rel_l2(got, ref, n) <= tol_any(n, 1, mixed=False)
    plan.execute(xd, out=xd)  # in place: a row's reads end before its writes begin
    assert np.array_equal(xd.cpu().numpy(), got)
    assert plan.status() == 0
    plan.close()
