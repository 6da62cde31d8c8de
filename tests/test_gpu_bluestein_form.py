"""Which Bluestein form a plan runs, as describe() names it, over every padded
length's default and the forms the environment selects (GPU); each default
against the FP64 oracle.

Bar: tests/helpers.py's Bluestein bound.
"""
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


@pytest.mark.parametrize("n", [17, 31, 37, 61, 67, 509, 1009, 2053, 4093, 8191, 8209])
def test_default_form(g, n):
    plan = g.Plan(n, 1, 3)
    d = plan.describe()["x"]
    M = d["bluestein_m"]
    assert M == bluestein_m(n) and d["half_q"] == (M // 2 if 128 <= M <= 16384 else 0)
    assert d["form"] == ("one_pass" if M < 128 else "half" if M <= 16384 else "five_pass")
    x = synth.uniform_complex((3, n), seed=n)
    got = plan.execute(torch.from_numpy(x).cuda()).cpu().numpy()
    ref = oracle.fft1d_any(x, dir=-1, threads=ORACLE_THREADS)
    assert worst_rel_l2(got, ref, n) <= tol_any(n, 1, mixed=False) and plan.status() == 0
    plan.close()


def test_selected_forms(g, monkeypatch):
    for name, value, form in (("ONEPASS", "1", "one_pass"), ("ONEPASS", "0", "two_pass"), ("FUSED", "0", "five_pass")):
        monkeypatch.setenv("GB300FFT_BLUESTEIN_" + name, value)
        plan = g.Plan(1009, 1, 3)
        d = plan.describe()
        assert (d["x"]["form"], d["x"]["half_q"], d["y"]["form"]) == (form, 0, "")
        plan.close()
        monkeypatch.delenv("GB300FFT_BLUESTEIN_" + name)
    plan = g.Plan(1000, 1, 1)
    assert plan.describe()["x"]["form"] == ""
    plan.close()
