"""Rates near 1 K: the product of the weights n''/w'' n'''/w''' of a term leaves FP64's range, while 1/n of the mode itself and the
rate in between are ordinary numbers.  One and several temperatures, FP64 and double-float, against a sum whose Bose factors
are one exponential per term."""
import numpy as np
import pytest

import oracle
from paper_2104_04895_gb300 import synth
from paper_2104_04895_gb300.binding import FP_PREC_DOUBLE_FLOAT, FP_PREC_FP64, Context

from conftest import oracle_modes

RTOL = 1e-10  # the FP64 bar of the library
HBAR, KB = 6.582119569e-4, 8.617333262e-5                  # eV ps, eV / K
CONV = 1.602176634e-19 / 1.66053906660e-27 * 1e-4          # eV / (A^2 amu) in ps^-2


def log_rates(cr, w, e, v, temps, window=2.0, sigma_min=1e-10):
    """Rates (nT, N nb) with the Bose factors of every term as one exponential, from the oracle's vertices: the
    product B / n overflows for no temperature at which a rate is a finite number."""
    N, nb, sb = cr.nq, cr.nb, cr.scalebroad
    grid = np.array(cr.grid)
    B = 2 * np.pi * np.linalg.inv(cr.lattice).T
    dq = np.cbrt(abs(np.linalg.det(B)) / N)
    G = np.stack(np.unravel_index(np.arange(N), cr.grid), 1)
    ok = w > 0.0
    out = np.zeros((len(temps), N, nb))
    with np.errstate(all="ignore"):
        x = HBAR * w[None] / (KB * np.asarray(temps)[:, None, None])
        ln = np.where(ok, -(x + np.log1p(-np.exp(-x))), 0.0)      # log n and log (1 + n)
        lp = np.where(ok, -np.log1p(-np.exp(-x)), 0.0)
    for q in range(N):
        for q1 in range(N):
            for q2 in range(N):
                for p, (s1, s2, c) in enumerate(((1, 1, 0.5), (1, -1, 0.5), (-1, -1, 1.0 / 6.0))):
                    V, q3 = oracle.v4(cr, e, q, q1, q2, p)
                    assert q3 == np.ravel_multi_index(tuple((G[q] + s1 * G[q1] + s2 * G[q2]) % grid), cr.grid)
                    W = [a.reshape([-1 if k == i else 1 for k in range(4)]) for i, a in
                         enumerate((w[q], w[q1], w[q2], w[q3]))]
                    dw = ((W[0] + s1 * W[1]) + s2 * W[2]) - W[3]
                    dv = v[q2][:, None, :] - v[q3][None, :, :]
                    sig = np.broadcast_to((sb * np.sqrt((dv ** 2).sum(-1)) * dq)[None, None], dw.shape)
                    use = np.abs(dw) <= window * np.maximum(sig, sigma_min)
                    for i, k in enumerate((q, q1, q2, q3)):
                        use = use & ok[k].reshape([-1 if n == i else 1 for n in range(4)])
                    if not use.any():
                        continue
                    a, b, g, d = np.nonzero(use)
                    s = sig[a, b, g, d]
                    small = s < sigma_min
                    s = np.where(small, 1.0, s)
                    delta = np.where(small, 1.0, np.exp(-(dw[a, b, g, d] / s) ** 2) / (np.sqrt(np.pi) * s))
                    f = c * np.abs(V[a, b, g, d]) ** 2 * delta / (w[q][a] * w[q1][b] * w[q2][g] * w[q3][d])
                    for t in range(len(temps)):
                        l1 = (lp if p < 2 else ln)[t, q1][b]
                        l2 = (lp if p < 1 else ln)[t, q2][g]
                        out[t, q] += np.bincount(a, f * np.exp(l1 + l2 + ln[t, q3][d] - ln[t, q][a]), nb)
    return (out * np.pi * HBAR ** 2 * CONV ** 4 / (8.0 * N * N)).reshape(len(temps), -1)


def _close(got, ref):
    """Rates below 1e-280 (none of interest) are left out: the terms of theirs need not be normal numbers."""
    use = ref > 1e-280
    assert use.sum() > 0.5 * ref.size
    assert np.max(np.abs(got[use] - ref[use]) / ref[use]) <= RTOL


@pytest.mark.parametrize("maker", [lambda: synth.simple_cubic((2, 2, 1)), lambda: synth.zincblende_bas((2, 1, 1))])
def test_reference_at_ordinary_temperatures(maker):
    cr = maker()
    w, e, v = oracle_modes(cr)
    ref, _ = oracle.rates4(cr, w, e, v, temps=[90.0, 300.0])
    mine = log_rates(cr, w, e, v, [90.0, 300.0])
    assert np.array_equal(ref == 0.0, mine == 0.0)
    assert np.max(np.abs(mine[ref > 0] - ref[ref > 0]) / ref[ref > 0]) <= 1e-11


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [FP_PREC_FP64, FP_PREC_DOUBLE_FLOAT])
@pytest.mark.parametrize("maker", [lambda: synth.simple_cubic((2, 2, 1)), lambda: synth.zincblende_bas((2, 1, 1)),
                                   lambda: synth.licoo2((1, 1, 1))])
def test_down_to_a_kelvin(precision, maker):
    """hbar w / k_B T of the highest mode from 100 to 600: 1/n is a normal number, the product of two n is not always.
    Mode tables given and the library's own."""
    cr = maker()
    with Context.from_crystal(cr) as ctx:
        for own in (True, False):
            if own:
                w, e, v = ctx.modes()
            else:
                w, e, v = oracle_modes(cr)
                ctx.set_modes(w, e, v)
            temps = [float(HBAR * w.max() / (KB * x)) for x in (100.0, 340.0, 450.0, 600.0)]
            ref = log_rates(cr, w, e, v, temps)
            out, _ = ctx.rates4(temps, cr.scalebroad, precision=precision)
            _close(out.reshape(len(temps), -1), ref)
            for t in range(len(temps)):
                one, _ = ctx.rates4(temps[t:t + 1], cr.scalebroad, precision=precision)
                _close(one.reshape(1, -1), ref[t:t + 1])
