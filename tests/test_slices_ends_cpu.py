"""CPU rebuild of the sliced contraction (fp_slices.cuh) at the ends of the digits' ranges: operands whose digits are all at
-256 or 255 under a top digit of 129 at most, where the level sums and the dropped levels are largest."""
from fractions import Fraction
from itertools import product

import numpy as np
import pytest

BIAS = sum(256 * 512 ** i for i in range(6))


def _digits(v):
    d = [(((v + BIAS) >> (9 * (5 - i))) & 511) - 256 for i in range(6)]
    assert sum(x * 512 ** (5 - i) for i, x in enumerate(d)) == v
    return d


def _value(d):
    return sum(x * 512 ** (5 - i) for i, x in enumerate(d))


@pytest.mark.parametrize("nb", [6, 12])
def test_level_sums_and_dropped_levels(nb):
    """Level sums below 2^24 (exact in FP32), below 2^22 where the kernel reads them from the low bits of a float, and the
    levels left out within 0.09 (six branches) and 0.19 (twelve) units of the last place."""
    bound = {6: 0.094, 12: 0.188}[nb]
    for ta, la, tb, lb in product((129, -129, 1), (-256, 255), (129, -129, 1), (-256, 255)):
        a, b = [ta] + [la] * 5, [tb] + [lb] * 5
        assert _digits(_value(a)) == a and _digits(_value(b)) == b
        K = 2 * nb
        D = [K * sum(a[i] * b[s - i] for i in range(6) if 0 <= s - i < 6) for s in range(11)]
        for s in range(7):
            assert float(np.float32(D[s])) == D[s] and abs(D[s]) < 2 ** 24
            if s < 5 and not (nb == 12 and s >= 3):
                assert abs(D[s]) < 2 ** 22
        dropped = Fraction(sum(D[s] * 512 ** (10 - s) for s in range(7, 11)), 2 ** 52)
        assert abs(dropped) <= bound
        assert sum(D[s] * 512 ** (10 - s) for s in range(11)) == K * _value(a) * _value(b)
