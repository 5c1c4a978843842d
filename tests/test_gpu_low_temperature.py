"""Rates at 10 and 20 K: the weights n''/w'' n'''/w''' of a term fall as exp(-hbar (w'' + w''') / k_B T), out of FP32's range
for the upper branches, while 1/n of the mode itself grows as fast; the rate in between stays an ordinary number.  One
and several temperatures, FP64 and double-float."""
import numpy as np
import pytest

import oracle
from paper_2104_04895_gb300 import synth
from paper_2104_04895_gb300.binding import FP_PREC_DOUBLE_FLOAT, FP_PREC_FP64, Context

from conftest import oracle_modes

RTOL = 1e-10  # the FP64 bar of the library


def _close(got, ref):
    zero = ref == 0.0
    assert np.all(got[zero] == 0.0)
    assert np.max(np.abs(got[~zero] - ref[~zero]) / ref[~zero]) <= RTOL


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [FP_PREC_FP64, FP_PREC_DOUBLE_FLOAT])
@pytest.mark.parametrize("maker", [lambda: synth.simple_cubic((3, 3, 2)), lambda: synth.diamond_si((3, 2, 2)),
                                   lambda: synth.zincblende_bas((3, 2, 2)), lambda: synth.licoo2((2, 2, 1))])
def test_ten_and_twenty_kelvin(precision, maker):
    cr = maker()
    w, e, v = oracle_modes(cr)
    temps = [10.0, 20.0, 300.0]
    ref, acc = oracle.rates4(cr, w, e, v, temps=temps)
    with Context.from_crystal(cr) as ctx:
        ctx.set_modes(w, e, v)
        out, st = ctx.rates4(temps, cr.scalebroad, precision=precision)
        _close(out.reshape(3, -1), ref)
        assert st["accepted"] == list(acc)
        for t in range(3):
            one, _ = ctx.rates4(temps[t:t + 1], cr.scalebroad, precision=precision)
            _close(one.reshape(1, -1), ref[t:t + 1])
        _, _, wp4 = ctx.phase_space4(temps, cr.scalebroad, precision=precision)
        ps, _ = oracle.rates4(cr, w, e, v, temps=temps, unit_vertex=True)
        _close(wp4.reshape(3, -1) * cr.nq ** 2, ps)
