"""Rounding of the Bluestein forms of padded lengths up to 16384, whose filter
spectra are built in FP64 (csrc/fft_bluestein.cu, k_filter64): relative L2 against
64 bits, Gaussian inputs.

Bound: the error of the length-M forms at these lengths with the filter transformed
in FP32, as measured over 2^23 points before the half-length form replaced them; it
moves by 0.3 % from one input to another.  The half-length form with that filter came
out up to 7 % above it at the shorter lengths.  The FP32 transform of the filter alone
is 0.9 to 1.3e-7 of it, its one rounding 0.3e-7.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LENGTH_M = {31: 1.603e-7, 61: 1.644e-7, 127: 2.060e-7, 251: 2.217e-7, 257: 1.759e-7, 509: 2.193e-7,
            1009: 2.324e-7, 2039: 2.583e-7, 4093: 2.778e-7, 4099: 2.244e-7, 8191: 2.743e-7}


@pytest.fixture(scope="module")
def g():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_15437_gb300 import build
    build.build()
    import paper_2506_15437_gb300 as g
    return g


@pytest.mark.parametrize("n", list(LENGTH_M))
@pytest.mark.parametrize("inverse", [False, True])
def test_no_further_than_the_length_m_forms(g, n, inverse):
    rows = (1 << 22) // n
    x = torch.randn(rows, n, dtype=torch.complex64, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(n))
    exact = x.to(torch.complex128)
    exact = torch.fft.ifft(exact, norm="forward") if inverse else torch.fft.fft(exact)
    plan = g.Plan(n, 1, rows, inverse=inverse)
    got = plan.execute(x).to(torch.complex128)
    assert float(torch.linalg.vector_norm(got - exact) / torch.linalg.vector_norm(exact)) <= 1.003 * LENGTH_M[n]
    plan.close()
