"""CPU rebuild of |W|^2 of a double-float complex (cdf_abs2, fp_rates_kernel.cuh) against exact rationals: the squares of the
low parts have one sign, so leaving them out would lower every rate by the same few 1e-16."""
from fractions import Fraction

import numpy as np

f32 = np.float32


def _fma(a, b, c):
    """FP32 fma: the product of two floats is exact in FP64; its sum with a third is rounded there and then to FP32."""
    return f32(np.float64(a) * np.float64(b) + np.float64(c))


def _abs2(xh, xl, yh, yl, low_squares):
    ph, qh = f32(xh * xh), f32(yh * yh)
    pe, qe = _fma(xh, xh, -ph), _fma(yh, yh, -qh)
    if low_squares:
        pe, qe = _fma(xl, xl, pe), _fma(yl, yl, qe)
    pe, qe = _fma(f32(2) * xh, xl, pe), _fma(f32(2) * yh, yl, qe)
    s = f32(ph + qh)
    bb = f32(s - ph)
    t = f32(f32(ph - f32(s - bb)) + f32(qh - bb))
    return float(np.float64(s) + np.float64(f32(t + f32(pe + qe))))


def test_no_common_bias():
    """A result is off by the FP32 roundings of its low part, 2^-23 of the result at most: a few 2^-47, with either sign, so
    that the mean of 4000 stays below 3 x 2^-47 / sqrt(4000) = 3.4e-16.  Without the low squares it is lower by their
    mean, some 2^-50 to 2^-48 of the result."""
    rng = np.random.default_rng(11)
    err = {True: [], False: []}
    for _ in range(4000):
        x, y = rng.normal(size=2)
        xh, yh = f32(x), f32(y)
        xl, yl = f32(x - float(xh)), f32(y - float(yh))
        exact = (Fraction(float(xh)) + Fraction(float(xl))) ** 2 + (Fraction(float(yh)) + Fraction(float(yl))) ** 2
        for k in err:
            err[k].append(float((Fraction(_abs2(xh, xl, yh, yl, k)) - exact) / exact))
    assert np.max(np.abs(err[True])) <= 4 * 2.0 ** -47
    assert abs(np.mean(err[True])) <= 3.4e-16
    assert np.mean(err[False]) < np.mean(err[True]) - 2.0 ** -51
