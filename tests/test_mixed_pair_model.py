"""CPU model of the in-place mixed-radix stages (csrc/fft_mixed_pair.cuh).

Every stage's butterflies are redone with the kernel's index arithmetic --
butterfly j to (p, q) and its place in the skewed buffer, the last stage's
digit reversal, the output position -- checking that they stay inside the
buffer, that each stage touches every element exactly once (so a butterfly may
overwrite what it read with no other one waiting for it) and that the result is
the DFT in natural order.
"""
import numpy as np
import pytest


def run(radix, skew):
    n, S = int(np.prod(radix)), len(radix)
    ns = [int(np.prod(radix[s + 1:])) for s in range(S)]
    kdiv = [int(np.prod(radix[1:s])) if s > 1 else 1 for s in range(S)]
    rng = np.random.Generator(np.random.PCG64(n + skew))
    x = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    buf = np.full(n + radix[0] * skew, np.nan + 0j)
    out = np.full(n, np.nan + 0j)
    for s, R in enumerate(radix):
        nb, Q = n // R, ns[s]
        D = np.exp(-2j * np.pi * np.outer(np.arange(R), np.arange(R)) / R)
        touched = np.zeros(buf.size, dtype=int)
        for j in range(nb):
            q, legs = j, np.arange(R)
            if s == 0:
                at = j + legs * (Q + skew)
            elif s == S - 1:
                rest, p, k0 = j, 0, 0
                for t in range(s):
                    rest, k = divmod(rest, radix[t])
                    k0 = k if t == 0 else k0
                    p = p * radix[t] + k
                at = p * R + k0 * skew + legs
            else:
                p, q = divmod(j, Q)
                at = p * R * Q + q + (p if s == 1 else p // kdiv[s]) * skew + legs * Q
            assert at.min() >= 0 and at.max() < buf.size
            touched[at] += 1
            v = D @ (x[j + legs * nb] if s == 0 else buf[at])
            if s == S - 1:
                out[j + legs * nb] = v
            else:
                buf[at] = v * np.exp(-2j * np.pi * legs * q / (R * Q))
        assert touched.max() == 1 and touched.sum() == n
    return np.linalg.norm(out - np.fft.fft(x)) / np.linalg.norm(x) / np.sqrt(n)


@pytest.mark.parametrize("radix", [(5, 3), (10, 10, 10), (12, 10, 9), (10, 6, 5, 10), (13, 5, 9, 7), (5, 4, 3, 2, 2)],
                         ids=str)
@pytest.mark.parametrize("skew", [0, 1, 3, 7])
def test_in_place_stages(radix, skew):
    assert run(list(radix), skew) < 1e-13
