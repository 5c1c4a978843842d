"""The mixed path's kernel for three and six branches where its bookkeeping can go wrong: one warp and several, idle
lanes, branch chunks, tiles of q', masks, single processes (each leaves other candidates to the compacted list), the
Normal and Umklapp parts, unit vertices, one temperature and the most."""
import numpy as np
import pytest

import oracle
from paper_2104_04895_gb300 import synth
from paper_2104_04895_gb300.binding import FP_PREC_MIXED, Context

from conftest import oracle_modes

pytestmark = pytest.mark.gpu

RTOL = 3e-6  # the mixed path's bound
# |W|^2 of an FP32 vertex that cancels: sums of some tens of terms, each rounded to 6e-8 of the largest, leave at most
# 1e-6 of it, and the square of that
NOISE = 1e-12


def _close(got, ref):
    assert np.all(got[ref == 0.0] <= NOISE * ref.max(initial=0.0))
    assert np.all(np.abs(got - ref) <= RTOL * ref + NOISE * ref.max(initial=0.0))


@pytest.mark.parametrize("maker,temps,opts", [
    (lambda: synth.simple_cubic((1, 1, 1)), [300.0], {}),
    (lambda: synth.simple_cubic((5, 3, 2)), [300.0], {}),
    (lambda: synth.simple_cubic((4, 3, 3)), list(np.linspace(250.0, 950.0, 8)), dict(block_j0=1, k1_tile=5)),
    (lambda: synth.diamond_si((2, 3, 2)), [300.0], {}),
    (lambda: synth.diamond_si((3, 2, 2)), [300.0, 700.0], dict(block_j0=2, threads=96)),
    (lambda: synth.zincblende_bas((3, 2, 3)), [400.0], dict(block_j0=1, threads=64, no_time_reversal=1)),
    (lambda: synth.zincblende_bas((3, 2, 2)), list(np.linspace(250.0, 950.0, 8)), {}),
])
def test_rates_masks_and_parts(maker, temps, opts):
    cr = maker()
    w, e, v = oracle_modes(cr)
    N, nb, nT = cr.nq, cr.nb, len(temps)
    rng = np.random.Generator(np.random.PCG64(N * nb + nT))
    run = dict(precision=FP_PREC_MIXED, **opts)
    with Context.from_crystal(cr) as ctx:
        ctx.set_modes(w, e, v)
        for mask in (None, (rng.random(N * nb) < 0.4).astype(np.uint8)):
            sel = np.arange(N * nb) if mask is None else np.nonzero(mask)[0]
            ref, acc = oracle.rates4(cr, w, e, v, temps=temps, sel=sel)
            out, st = ctx.rates4(temps, cr.scalebroad, mode_mask=mask, **run)
            flat = out.reshape(nT, -1)
            _close(flat[:, sel], ref)
            assert np.all(np.delete(flat, sel, axis=1) == 0.0)
            assert st["accepted"] == list(acc)
            again, _ = ctx.rates4(temps, cr.scalebroad, mode_mask=mask, **run)
            assert np.array_equal(out, again)
        for p in range(3):
            ref, acc = oracle.rates4(cr, w, e, v, temps=temps, processes=(p,))
            out, st = ctx.rates4(temps, cr.scalebroad, process_mask=1 << p, **run)
            _close(out.reshape(nT, -1), ref)
            assert st["accepted"][p] == acc[p]
        for s, name in ((1, "normal"), (2, "umklapp")):
            ref, acc = oracle.rates4(cr, w, e, v, temps=temps, nu=name)
            out, st = ctx.rates4(temps, cr.scalebroad, nu_select=s, **run)
            _close(out.reshape(nT, -1), ref)
            assert st["accepted"] == list(acc)
        npr, _, wp4 = ctx.phase_space4(temps, cr.scalebroad, **run)
        ref, acc = oracle.rates4(cr, w, e, v, temps=temps, unit_vertex=True)
        _close(wp4.reshape(nT, -1) * N ** 2, ref)
        assert npr.sum() == acc.sum()
