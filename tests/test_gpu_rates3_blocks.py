"""fp_rates3 where its launch can go wrong: k1 ranges with a remainder, more temperatures than the shared memory holds
Psi beside, masks that select one member of a pair {q, -q}, points that are their own -q, and a wide window (Gaussian
arguments beyond its table)."""
import numpy as np
import pytest

import oracle
from paper_2104_04895_gb300 import synth
from paper_2104_04895_gb300.binding import Context

from conftest import oracle_modes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("maker,nT,window", [
    (lambda: synth.simple_cubic((5, 3, 2)), 1, 2.0), (lambda: synth.simple_cubic((2, 2, 2)), 8, 3.0),
    (lambda: synth.diamond_si((5, 2, 3)), 3, 2.0), (lambda: synth.zincblende_bas((1, 4, 5)), 1, 2.5),
    (lambda: synth.licoo2((3, 2, 1)), 8, 2.0), (lambda: synth.licoo2((1, 1, 1)), 1, 2.0)])
def test_rates3_blocks(maker, nT, window):
    cr = maker()
    w, e, v = oracle_modes(cr)
    N, nb = cr.nq, cr.nb
    temps = list(np.linspace(250.0, 900.0, nT))
    rng = np.random.Generator(np.random.PCG64(N))
    with Context.from_crystal(cr) as ctx:
        ctx.set_modes(w, e, v)
        for mask in (None, (rng.random(N * nb) < 0.3).astype(np.uint8)):
            sel = np.arange(N * nb) if mask is None else np.nonzero(mask)[0]
            ref, acc = oracle.rates3(cr, w, e, v, temps=temps, sel=sel, window=window)
            out, st = ctx.rates3(temps, cr.scalebroad, mode_mask=mask, window=window)
            got = out.reshape(nT, -1)[:, sel]
            zero = ref == 0.0
            assert np.all(got[zero] == 0.0)
            # terms of the + process change sign with n' - n'', so the bound is relative to the sum of magnitudes
            assert np.max(np.abs(got - ref)) <= 1e-10 * np.max(np.abs(ref), initial=0.0)
            # relative where the vertex does not vanish by symmetry (there both sides hold rounding, 1e-30 and below)
            live = np.abs(ref) > 1e-20 * np.max(np.abs(ref), initial=0.0)
            assert np.max(np.abs(got[live] - ref[live]) / np.abs(ref[live]), initial=0.0) <= 1e-9
            assert np.all(np.delete(out.reshape(nT, -1), sel, axis=1) == 0.0)
            assert st["accepted"][:2] == list(acc)
