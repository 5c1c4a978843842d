"""Device memory of the rate calls: a call whose fastest form finds no memory takes a smaller form instead of failing, and
large working memory is given back with the call.  Failing allocations are injected on the host (FP_FAULT_ALLOC)."""
import numpy as np
import pytest

from paper_2104_04895_gb300 import synth
from paper_2104_04895_gb300.binding import FP_PREC_DOUBLE_FLOAT, FP_PREC_FP64, FP_PREC_MIXED, Context

pytestmark = pytest.mark.gpu


def _close(got, ref, tol):
    big = ref > 0
    assert np.all(got[~big] == 0.0)
    assert np.max(np.abs(got - ref)[big] / ref[big]) <= tol


@pytest.mark.parametrize("precision", [FP_PREC_FP64, FP_PREC_DOUBLE_FLOAT, FP_PREC_MIXED])
@pytest.mark.parametrize("maker", [lambda: synth.simple_cubic((4, 3, 3)), lambda: synth.diamond_si((3, 3, 2)),
                                   lambda: synth.licoo2((2, 2, 1))])
def test_a_call_that_finds_no_memory_takes_a_smaller_form(maker, precision, monkeypatch):
    """The second allocation of a first call is its working memory; the parts and the phase space allocate likewise."""
    cr = maker()
    temps = [300.0, 700.0]
    calls = {"rates4": lambda c: c.rates4(temps, cr.scalebroad, precision=precision),
             "nu": lambda c: c.rates4_nu(temps, cr.scalebroad, precision=precision),
             "channels": lambda c: c.rates4_channels(temps, cr.scalebroad, precision=precision),
             "phase": lambda c: c.phase_space4(temps, cr.scalebroad, precision=precision)}
    # the mixed kernels' sums differ by their order and rounding
    tol = 1e-6 if precision == FP_PREC_MIXED else 1e-12
    for name, call in calls.items():
        res = []
        for fault in (False, True):
            with Context.from_crystal(cr) as ctx:
                ctx.modes(copy=False)
                if fault:
                    monkeypatch.setenv("FP_FAULT_ALLOC", "2")
                res.append(call(ctx))
                if fault:
                    monkeypatch.delenv("FP_FAULT_ALLOC")
        if name == "phase":
            for a, b in zip(res[1], res[0]):
                _close(a, b, tol)
            continue
        (ref, st), (got, st2) = res
        big = ref > 1e-20 * ref.max()  # the parts may hold rates that vanish by symmetry
        assert np.max(np.abs(got - ref)[big] / ref[big]) <= tol
        assert st["accepted"] == st2["accepted"]
        if name == "rates4" and precision != FP_PREC_MIXED:
            assert st2["terms_executed"] > 1.2 * st["terms_executed"]  # every q' evaluated, not each pair once


def test_large_working_memory_is_given_back():
    """Simple cubic 12x12x11 with eight temperatures: 242 MB of slots, one per pair and temperature."""
    import torch
    cr = synth.simple_cubic((12, 12, 11))
    temps = list(np.linspace(300.0, 1000.0, 8))
    one = np.zeros(cr.nq * cr.nb, np.uint8)
    one[7] = 1
    with Context.from_crystal(cr) as ctx:
        ctx.modes(copy=False)
        ctx.rates4(temps, cr.scalebroad, mode_mask=one)
        free = torch.cuda.mem_get_info()[0]
        first, _ = ctx.rates4(temps, cr.scalebroad)
        assert torch.cuda.mem_get_info()[0] > free - (64 << 20)
        again, _ = ctx.rates4(temps, cr.scalebroad)
    assert np.array_equal(first, again)


def test_phase_space_over_ordered_sums():
    """The form of last resort, which force constants without the leg symmetry take too: the phase space does not see them."""
    cr = synth.zincblende_bas((3, 2, 2))
    temps = [300.0, 500.0, 700.0]
    rng = np.random.Generator(np.random.PCG64(5))
    with Context.from_crystal(cr) as ctx:
        ctx.modes(copy=False)
        ref = ctx.phase_space4(temps, cr.scalebroad)
    cr.fc4_val = cr.fc4_val + rng.normal(0.0, 1.0, cr.fc4_val.shape)
    with Context.from_crystal(cr) as ctx:
        ctx.modes(copy=False)
        got = ctx.phase_space4(temps, cr.scalebroad)
    for a, b in zip(got, ref):
        _close(a, b, 1e-12)
