"""CPU rebuild of the sliced contraction (fp_slices.cuh): fixed point, balanced digits, exact level sums and their
combination, in integers, against exact rationals."""
from fractions import Fraction

import numpy as np
import pytest

BIAS = sum(256 * 512 ** i for i in range(6))


def _digits(v):
    d = [(((v + BIAS) >> (9 * (5 - i))) & 511) - 256 for i in range(6)]
    assert sum(x * 512 ** (5 - i) for i, x in enumerate(d)) == v
    return d


@pytest.mark.parametrize("nb", [6, 12])
def test_product_within_the_rounding_of_the_scale(nb):
    """|error| <= 4 2^-53 of the scale: 1/2 unit of 2^-52 from the result, at most sqrt(2 nb) / 2 units from the operands
    (each off by 1/2 unit, the other one of norm at most 1), 1/16 from the levels left out; rms near one unit of 2^-53."""
    rng = np.random.default_rng(nb)
    errs = []
    for _ in range(200):
        a = rng.normal(size=2 * nb) * 10.0 ** rng.uniform(-3, 3)
        e = rng.normal(size=2 * nb)
        e /= np.linalg.norm(e)
        s = int(np.floor(np.log2(np.linalg.norm(a) * 1.0001))) + 1
        fa = [_digits(round(Fraction(x) * 2 ** 52 / Fraction(2) ** s)) for x in a]
        fe = [_digits(round(Fraction(x) * 2 ** 52)) for x in e]
        D = [sum(x[i] * y[l - i] for x, y in zip(fa, fe) for i in range(6) if 0 <= l - i < 6) for l in range(7)]
        q = np.float32(D[6]) * np.float32(1 / 512) + np.float32(D[5])
        T = int(np.rint(float(q) / 128)) + sum(D[l] * 2 ** (38 - 9 * l) for l in range(5))
        exact = sum(Fraction(x) * Fraction(y) for x, y in zip(a, e)) / Fraction(2) ** s
        errs.append(float((Fraction(T, 2 ** 52) - exact) * 2 ** 53))
    assert np.max(np.abs(errs)) <= 1.0 + np.sqrt(2 * nb) + 0.125 + 1.0
    assert np.sqrt(np.mean(np.square(errs))) <= 1.5


@pytest.mark.parametrize("nb", [6, 12])
def test_level_sums_stay_exact_integers(nb):
    """Bounds of |D_s| from the digit ranges (top digit at most 129, the others 256): below 2^24, so that FP32 holds
    them exactly, and below 2^22 where the kernel reads them from the low bits of float + 1.5 2^23."""
    top = [129] + [256] * 5
    for s in range(7):
        bound = 2 * nb * sum(top[i] * top[s - i] for i in range(6) if 0 <= s - i < 6)
        assert bound < 2 ** 24
        if not (nb == 12 and s >= 3) and s < 5:
            assert bound < 2 ** 22


def test_range_ends():
    for v in (-(2 ** 52) - 2 ** 20, -(2 ** 52), -1, 0, 1, 2 ** 52, 2 ** 52 + 2 ** 20):
        d = _digits(v)
        assert abs(d[0]) <= 129 and all(-256 <= x <= 255 for x in d)
