"""The allocation kernel's short expm1 series: below 2^-3 it starts the Horner scheme at x^9
instead of x^16, which must not change a bit of the result."""
import math

import numpy as np
import pytest

E1 = [np.float32(0)] + [np.float32(1.0 / math.factorial(k)) for k in range(1, 17)]


def horner(x, m):
    p = np.full_like(x, E1[m])
    for k in range(m - 1, 0, -1):
        p = p * x + E1[k]          # float32: each operation rounded once
    return p * x


@pytest.mark.parametrize("e", [-3, -4, -5, -6, -8, -12, -20, -60, -126])
def test_short_series_is_bit_exact(e):
    """Every float of the binade [2^(e-1), 2^e) (every 64th below 2^-6)."""
    step = 1 if e >= -6 else 64
    for part in range(8):
        bits = np.arange(part << 20, (part + 1) << 20, step, dtype=np.uint32) + np.uint32((127 + e - 1) << 23)
        x = bits.view(np.float32)
        assert np.array_equal(horner(x, 16), horner(x, 9))


def test_series_is_the_oracles(orc):
    for x in np.float32([0.12, 0.11, 1e-2, 3e-3, 1e-5]):
        assert np.float32(orc.expm1_series(float(x))) == horner(np.array([x]), 9)[0]


@pytest.mark.timeout(60, method="thread")
def test_series_of_an_infinite_argument(orc):
    """An erasure statistic that overflowed (|k|^2 beyond FP32's range): the halving must end.  expm1 is
    infinite, and so from about 89 on."""
    for x in (np.inf, np.finfo(np.float32).max, 1e30, 200.0):
        assert orc.expm1_series(float(np.float32(x))) == np.inf
    assert orc.expm1_series(float("nan")) == 0.0 and orc.expm1_series(float("-inf")) == 0.0
