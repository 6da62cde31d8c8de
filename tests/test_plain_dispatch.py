"""When fft1 / fft2 may call the plan directly (host logic, no GPU): never where
an autograd Function would have recorded, transformed or refused the call."""
import torch
from torch.autograd import forward_ad

from paper_2506_15437_gb300 import fft


def test_plain_only_where_a_function_would_do_nothing():
    x = torch.zeros(4, 4, dtype=torch.complex64)
    assert fft._plain(x)
    w = x.clone().requires_grad_(True)
    assert not fft._plain(w)
    with torch.no_grad():
        assert fft._plain(w)
    with torch.inference_mode():
        assert fft._plain(x)
    assert not fft._plain(torch.nn.Parameter(x))  # a subclass
    assert not fft._plain([1, 2])
    with forward_ad.dual_level():
        assert not fft._plain(x) and not fft._plain(forward_ad.make_dual(x, x))
    assert fft._plain(x)


def test_not_plain_under_transforms_and_tracing():
    seen = []

    def f(x):
        seen.append(fft._plain(x))
        return x * 2

    x = torch.zeros(3, 4)
    torch.func.vmap(f)(x)
    torch.func.jvp(f, (x,), (x,))
    torch.func.grad(lambda t: f(t).sum())(x)
    torch.jit.trace(f, x, check_trace=False)
    assert len(seen) >= 4 and not any(seen)
