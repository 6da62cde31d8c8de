"""Lazily conjugated and negated tensors (x.conj(), the imaginary part of one)
reach the library as the values they stand for (host logic, no GPU): a
stand-in library copies the memory it is given, so an unresolved view shows as
its unconjugated values.
"""
import ctypes

import pytest
import torch

from paper_2506_15437_gb300 import fft


class CopyLib:
    """The entry points used here as copies of the raw memory they are given."""

    def __init__(self, n):
        self.n = n

    def fft_execute(self, p, x, out, stream):
        ctypes.memmove(out, x, 8 * self.n)
        return 0

    def fft_backward(self, p, g, out, stream):
        return self.fft_execute(p, g, out, stream)

    def fft_execute_host(self, p, x, out, stream):
        return self.fft_execute(p, x, out, stream)

    def fft_weighted_power_adjoint_parts(self, p):
        return 1

    def fft_weighted_power_adjoint(self, p, x, w, partials, y, stream):
        ctypes.memmove(partials, w, 4)
        return self.fft_execute(p, x, y, stream)

    def fft_backward_rows_scaled(self, p, y, scale_dev, scale, out, stream):
        self.scale = ctypes.c_float.from_address(scale_dev).value
        return self.fft_execute(p, y, out, stream)

    def fft_plan_destroy(self, p):
        pass


@pytest.fixture
def plan(monkeypatch):
    n = 12
    p = fft.Plan.__new__(fft.Plan)
    p.nx, p.ny, p.batch, p._p, p._lib = 4, 3, 1, 1, CopyLib(n)

    def check(t, dtype, name):  # as fft._check_tensor, for CPU tensors
        assert t.dtype == dtype and t.is_contiguous()

    monkeypatch.setattr(fft, "_check_tensor", check)
    monkeypatch.setattr(fft, "_stream_handle", lambda device: 0)
    monkeypatch.setattr(fft, "_raw_stream", lambda index: 0, raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda index: 0, raising=False)
    monkeypatch.setattr(fft, "get_plan", lambda *a: p)
    return p


def data():
    return torch.randn(3, 4, dtype=torch.complex64, generator=torch.Generator().manual_seed(5))


VIEWS = {"conj": lambda x: x.conj(), "neg": torch._neg_view, "both": lambda x: torch._neg_view(x.conj())}


@pytest.mark.parametrize("view", VIEWS)
def test_inputs(plan, view):
    v = VIEWS[view](data())
    want = v.clone()
    assert (v.is_conj() or v.is_neg()) and v.contiguous().data_ptr() == v.data_ptr()
    for call in (fft.fft2, fft.fft1, plan.execute, plan.backward, lambda t: plan.backward_rows_scaled(t, torch.ones(1))):
        got = call(v)
        assert torch.equal(got, want) and not got.is_conj() and not got.is_neg()
    with pytest.raises(ValueError):
        plan.execute(data(), out=v)


def test_host_calls(plan, monkeypatch):
    synced = []
    monkeypatch.setattr(torch.cuda, "current_stream",
                        lambda dev=None: type("S", (), {"synchronize": lambda self: synced.append(1)})())
    x = data()
    assert torch.equal(plan.execute_host(x), x) and not synced
    assert torch.equal(plan.execute_host(x.conj()), x.conj().clone()) and synced
    with pytest.raises(ValueError):
        plan.execute_host(x, out=data().conj())


def test_gradients(plan):
    x, c = data().requires_grad_(True), data()
    for f in (fft.fft2, fft.fft1):
        (g,) = torch.autograd.grad((f(x).conj() * c).real.sum(), x)
        # the stand-in is the identity: the gradient of Re sum conj(x) c is conj(conj(c))
        assert torch.equal(g.resolve_conj(), c)


def test_loss(plan):
    x = data().requires_grad_(True)
    w = torch._neg_view(torch.full((3, 4), -2.0))
    assert w.is_neg()
    loss = fft.weighted_power_loss(x.conj(), w)
    assert loss.item() == 2.0  # the stand-in's loss is w[0]
    loss.backward(torch._neg_view(torch.tensor(-3.0)))
    assert plan._lib.scale == 3.0
