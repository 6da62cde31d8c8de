"""The mixed-radix launches plans make (fft_debug_mixed_launch, host only),
over row, column and four-step passes, small and large: the stages are a
schedule of the length in the fewest stages, the CTA fits the hardware, and the
kernel's index arithmetic over that schedule and skew -- redone by
test_mixed_pair_model.py's model -- gives the DFT; its twiddle tables hold every
factor once, at the pair the stage reads.
"""
import ctypes

import numpy as np
import pytest

from tests.test_abi import MIXED_RADICES, _fewest_stages, _smooth13
from tests.test_mixed_pair_model import run

MAX_SMEM = 227 * 1024


@pytest.fixture(scope="module")
def lib():
    from paper_2506_15437_gb300 import build
    build.build()
    from paper_2506_15437_gb300 import _native as N
    return N.load()


def launch(lib, n, nx=0, count=1, fourstep=0, n1=0):
    info = (ctypes.c_int * 24)()
    assert lib.fft_debug_mixed_launch(n, nx, count, fourstep, n1, info) == 0, (n, nx, count, fourstep, n1)
    keys = ("lanes", "W", "threads", "smem", "rmax", "skew", "buf", "S")
    d = dict(zip(keys, info))
    d["radix"] = list(info[8:8 + d["S"]])
    assert not any(info[8 + d["S"]:])
    return d


# (nx, count, fourstep, n1): rows few and many, columns even and odd, the passes of a four-step transform
LAYOUTS = [(0, 1, 0, 0), (0, 37, 0, 0), (0, 1 << 20, 0, 0), (1080, 1080 << 8, 0, 0), (1081, 1081 << 8, 0, 0),
           (6, 6, 0, 0), (120, 120, 1, 0), (0, 120, 1, 120), (0, 1000 * 32, 1, 1000)]


def test_schedules_and_limits(lib):
    fewest = _fewest_stages(14336)
    for n in [m for m in range(2, 1200) if _smooth13(m)] + [1728, 3000, 4095, 6000, 7000, 7168, 10000, 14300, 14336]:
        for lay in LAYOUTS:
            d = launch(lib, n, *lay)
            key = (n, lay, d)
            assert int(np.prod(d["radix"])) == n and set(d["radix"]) <= MIXED_RADICES, key
            split = fewest[n] == 1 and n >= 8 and n not in (11, 13)  # one stage reads and writes rows uncoalesced
            assert d["S"] == (2 if split else fewest[n]) <= 16, key
            assert max(d["radix"]) <= d["rmax"], key
            assert d["buf"] == n + d["radix"][0] * d["skew"] and 0 <= d["skew"] < 8, key
            words = d["W"] // d["lanes"]
            assert d["W"] == words * d["lanes"] and d["smem"] == words * d["buf"] * 8 * d["lanes"] <= MAX_SMEM, key
            limit = 1024 if d["lanes"] == 1 else 640 if d["rmax"] == 13 else 512
            assert d["threads"] % 32 == 0 and 32 <= d["threads"] <= limit, key
            nx, count, fourstep, n1 = lay
            if nx or n1:  # transforms taken fastest: shifts and masks
                assert words & (words - 1) == 0, key
            if fourstep or nx % 2 or n > 7000:
                assert d["lanes"] == 1, key
    # both forms, and both classes of the one over pairs, are in the table
    seen = {(launch(lib, n, *lay)["lanes"], launch(lib, n, *lay)["rmax"]) for n in (100, 210, 1000) for lay in LAYOUTS}
    assert seen == {(1, 16), (2, 13), (2, 16)}


@pytest.mark.parametrize("n", [8, 15, 96, 100, 384, 1000, 1080, 1920, 2197, 3000, 4095, 14336])
@pytest.mark.parametrize("lay", LAYOUTS, ids=str)
def test_index_arithmetic(lib, n, lay):
    d = launch(lib, n, *lay)
    if len(d["radix"]) == 1:
        pytest.skip("one stage: no buffer")
    assert run(d["radix"], d["skew"]) < 1e-13


@pytest.mark.parametrize("n", [7, 96, 1000, 1728, 2197, 4095])
@pytest.mark.parametrize("lay", [LAYOUTS[0], LAYOUTS[2], LAYOUTS[3]], ids=str)
def test_twiddle_tables(lib, n, lay):
    radix = launch(lib, n, *lay)["radix"]
    Q = n
    for R in radix:
        Q //= R  # product of the radices after the stage
        stride = R & ~1  # R - 1 rounded up to even
        e = np.arange(Q * stride)
        pair, odd = e >> 1, e & 1
        p, k = pair // Q, pair % Q
        r = 2 * p + 1 + odd
        real = r < R
        assert len(set(zip(k[real].tolist(), r[real].tolist()))) == real.sum() == Q * (R - 1)
        # the stage reads twiddles r, r + 1 of butterfly q at 16-byte pair (r - 1) / 2 * Q + q
        q, rr = np.meshgrid(np.arange(Q), np.arange(1, R, 2))
        at = 2 * ((rr - 1) // 2 * Q + q)
        assert at.max() + 1 < e.size
        assert np.array_equal(k[at], q) and np.array_equal(r[at], rr) and np.array_equal(r[at + 1], rr + 1)
    assert Q == 1


def test_refusals(lib):
    info = (ctypes.c_int * 24)()
    for n in (0, 1, 17, 14337, 2 * 14336):
        assert lib.fft_debug_mixed_launch(n, 0, 1, 0, 0, info) == -1
    for args in ((8, -1, 1, 0, 0), (8, 0, 0, 0, 0), (8, 8, 8, 1, 4), (8, 0, 1, 1, -1)):
        assert lib.fft_debug_mixed_launch(*args, info) == -2, args
    assert lib.fft_debug_mixed_launch(8, 0, 1, 0, 0, None) == -2
