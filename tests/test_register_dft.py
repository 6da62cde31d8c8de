"""The 32- and 64-point register DFTs (csrc/fft_common.cuh, dif_level4): a model
of their radix-4 levels, and the rounding of the passes built on them.

A transform in 32- and 64-point stages has one exchange where 16-point stages
have two, but radix-2 levels rotate half the values at each of more levels, and
every rotation rounds: 1024 points as 32 x 32 came out 5 % further from the exact
result than as 4 x 16 x 16.  Levels of radix 4 rotate a value at most once in two
levels.  The bound below is the error of the same lengths in stages of at most
16 points, emulated in float32 with fused multiply-adds and twiddles rounded once
(relative L2, Gaussian inputs, 2^19 points; its spread there is 0.1 %); from 1024
points the 32- and 64-point stages are emulated 1.0 to 3.5 % below it with radix 4
and 1.5 to 5.6 % above it with radix 2.  512 = 16 x 32 is on it with radix 2, which
its kernels keep.
"""
import numpy as np
import pytest

STAGES_OF_16 = {512: 1.096e-7, 1024: 1.141e-7, 2048: 1.202e-7, 4096: 1.292e-7}


def bitrev(k, bits):
    return int(format(k, f"0{bits}b")[::-1], 2) if bits else 0


def level2(a, H):
    for blk in range(0, len(a), 2 * H):
        for k in range(H):
            u, v = a[blk + k].copy(), a[blk + k + H].copy()
            a[blk + k], a[blk + k + H] = u + v, (u - v) * np.exp(-2j * np.pi * k * (64 // (2 * H)) / 64)


def dft(x):
    """dft<R> as the kernels run it: dif_level4 from span R / 4, a last odd level of radix 2."""
    a, R = x.astype(complex), len(x)
    Q, rotations = R // 4, 0
    while Q >= 1:
        U = 16 // Q
        for blk in range(0, R, 4 * Q):
            for k in range(Q):
                p = [blk + k + i * Q for i in range(4)]
                s02, d02, s13, d13 = a[p[0]] + a[p[2]], a[p[0]] - a[p[2]], a[p[1]] + a[p[3]], a[p[1]] - a[p[3]]
                for at, v, q in ((p[0], s02 + s13, 0), (p[1], s02 - s13, 2 * k * U), (p[2], d02 - 1j * d13, k * U),
                                 (p[3], d02 + 1j * d13, 3 * k * U)):
                    assert 0 <= q < 48 and (at == p[1] or q == 0 or q % 16)  # the forms mul_root64 has for pairs
                    rotations += q % 16 != 0
                    a[at] = v * np.exp(-2j * np.pi * q / 64)
        if Q == 2:
            level2(a, 1)
            break
        Q //= 4
    return a[[bitrev(k, R.bit_length() - 1) for k in range(R)]], rotations / R


@pytest.mark.parametrize("R,per_point", [(16, 0.5), (32, 0.875), (64, 1.1875)])
def test_levels_are_the_dft(R, per_point):
    rng = np.random.Generator(np.random.PCG64(R))
    x = rng.standard_normal((R, 5)) + 1j * rng.standard_normal((R, 5))
    y, rotations = dft(x)
    assert np.abs(y - np.fft.fft(x, axis=0)).max() < 1e-13
    assert rotations == per_point  # radix-2 levels: 0.625, 1.0625, 1.53125


@pytest.fixture(scope="module")
def g():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_15437_gb300 import build
    build.build()
    import paper_2506_15437_gb300 as g
    return g


def error(plan, x, dim):
    import torch
    ref = torch.fft.fft(x.cdouble(), dim=dim)
    return (torch.linalg.norm(plan.execute(x) - ref) / torch.linalg.norm(ref)).item()


def gaussian(*shape):
    import torch
    return torch.randn(*shape, dtype=torch.complex64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(7))


@pytest.mark.gpu
@pytest.mark.parametrize("n,e", [(512, 32), (1024, 32), (2048, 64), (4096, 64)])
def test_column_rounding(g, n, e):
    from paper_2506_15437_gb300.fft import ColumnPlan
    plan = ColumnPlan(1024, n, 8)
    assert plan.describe()["cols"]["e"] == e
    assert error(plan, gaussian(8, n, 1024), -2) <= STAGES_OF_16[n]
    plan.close()


@pytest.mark.gpu
@pytest.mark.parametrize("n", [512, 1024, 4096])
def test_row_rounding(g, n):
    plan = g.Plan(n, 1, (1 << 24) // n)
    assert plan.describe()["rows"]["e"] == 32
    assert error(plan, gaussian((1 << 24) // n, n), -1) <= STAGES_OF_16[n]
    plan.close()
