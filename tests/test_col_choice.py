"""What the column pass runs and what the autotuner times beside it
(fft_debug_col_choice, host only): every compiled number of elements per
thread is either the plan's choice or a candidate, on both sides of the rule
that takes 16 where the tiles are too few to fill the SMs.
"""
import ctypes

import pytest

SMS = 152
# elements per thread compiled for a column length
COMPILED = {32: [16], 64: [16], 128: [16], 256: [16], 512: [16, 32], 1024: [16, 32], 2048: [16, 64], 4096: [16, 32, 64],
            8192: [16, 32, 64]}


@pytest.fixture(scope="module")
def lib():
    from paper_2506_15437_gb300 import build
    build.build()
    from paper_2506_15437_gb300 import _native as N
    return N.load()


def choice(lib, n, nx, batch):
    info = (ctypes.c_int * 6)()
    assert lib.fft_debug_col_choice(n, nx, batch, SMS, info) == 0
    assert not any(info[3 + info[2]:])
    return info[0], info[1], list(info[3:3 + info[2]])


@pytest.mark.parametrize("n", COMPILED)
@pytest.mark.parametrize("nx,batch", [(2, 1), (4, 1), (64, 1), (512, 1), (1024, 1), (512, 64), (1024, 16), (8192, 1)])
def test_every_variant_is_chosen_or_timed(lib, n, nx, batch):
    e, w, others = choice(lib, n, nx, batch)
    assert w <= nx and n * w <= 16384
    assert sorted([e, *others]) == COMPILED[n]
    if n in (512, 1024, 2048):
        few = nx * batch / w < SMS
        assert e == (16 if few else COMPILED[n][-1])
        assert (w <= 4) if few else True


def test_short_columns_and_refusals(lib):
    for n in (2, 4, 8):
        e, _, others = choice(lib, n, 64, 1)
        assert e == n and others == []
    info = (ctypes.c_int * 6)()
    for bad in ((1, 64, 1, SMS), (48, 64, 1, SMS), (16384, 64, 1, SMS), (512, 1, 1, SMS), (512, 48, 1, SMS)):
        assert lib.fft_debug_col_choice(*bad, info) == -1, bad
    for bad in ((512, 64, 0, SMS), (512, 64, 1, 0)):
        assert lib.fft_debug_col_choice(*bad, info) == -2, bad
    assert lib.fft_debug_col_choice(512, 64, 1, SMS, None) == -2
