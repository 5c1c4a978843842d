"""The tiles of the kernel over pairs: the tile that a call reports can be asked for, up to the widest block (two branches of
twelve in nine warps), and a tuned context is no slower than an untuned one."""
import numpy as np
import pytest

from paper_2104_04895_gb300 import synth
from paper_2104_04895_gb300.binding import (FP_EINVAL, FP_PREC_DOUBLE_FLOAT, FP_PREC_FP64, FP_PREC_MIXED, Context,
                                            FourPhononError)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [FP_PREC_FP64, FP_PREC_DOUBLE_FLOAT])
@pytest.mark.parametrize("temps", [[300.0], [300.0, 700.0]])
def test_reported_tile_replays(precision, temps):
    cr = synth.licoo2((3, 2, 1))
    with Context.from_crystal(cr) as ctx:
        ctx.modes(copy=False)
        auto, st = ctx.rates4(temps, cr.scalebroad, precision=precision)
        j, t1, th, _ = st["tile"]
        assert (j, th) == (2, 288)
        same, st2 = ctx.rates4(temps, cr.scalebroad, precision=precision, block_j0=j, k1_tile=t1, threads=th)
        assert st2["tile"][:3] == st["tile"][:3] and np.array_equal(auto, same)
        for bad in (dict(block_j0=2, threads=256), dict(block_j0=2, threads=320), dict(block_j0=3),
                    dict(block_j0=5), dict(block_j0=1, threads=150)):
            with pytest.raises(FourPhononError) as ei:
                ctx.rates4(temps, cr.scalebroad, precision=precision, **bad)
            assert ei.value.code == FP_EINVAL
        # the kernel over ordered sums, which runs this path, has no such tile
        with pytest.raises(FourPhononError) as ei:
            ctx.rates4(temps, cr.scalebroad, precision=FP_PREC_MIXED, block_j0=2)
        assert ei.value.code == FP_EINVAL and "160" in str(ei.value)


@pytest.mark.parametrize("precision,maker", [(FP_PREC_FP64, lambda: synth.licoo2((5, 4, 3))),
                                             (FP_PREC_DOUBLE_FLOAT, lambda: synth.licoo2((3, 3, 2))),
                                             (FP_PREC_FP64, lambda: synth.diamond_si((4, 4, 4))),
                                             (FP_PREC_MIXED, lambda: synth.diamond_si((4, 4, 4)))])
def test_a_tuned_context_is_not_slower(precision, maker):
    cr = maker()
    with Context.from_crystal(cr) as ctx:
        ctx.modes(copy=False)

        def run():
            got = [ctx.rates4(cr.temps, cr.scalebroad, precision=precision) for _ in range(6)]
            return got[0][0], min(st["ms"] for _, st in got[1:]), got[0][1]

        out, ms, st = run()
        tiles, best = ctx.autotune(cr.temps, cr.scalebroad, precision=precision)
        tuned, ms_tuned, st_tuned = run()
        assert [tiles[k] for k in ("block_j0", "k1_tile", "threads")] == st_tuned["tile"][:3]
        assert ms_tuned <= 1.10 * ms and best > 0.0
        assert st_tuned["accepted"] == st["accepted"]
        big = out > 0
        tol = 1e-9 if precision == FP_PREC_MIXED else 1e-12  # the order of the sums
        assert np.max(np.abs(tuned - out)[big] / out[big]) <= tol


def test_a_tile_tuned_for_few_sums_leaves_the_others_valid():
    cr = synth.licoo2((3, 2, 1))
    temps = list(np.linspace(300.0, 1000.0, 8))
    with Context.from_crystal(cr) as ctx:
        ctx.modes(copy=False)
        ref, st = ctx.rates4(temps, cr.scalebroad)
        ctx.autotune(temps[:2], cr.scalebroad)
        ctx.autotune(temps[:1], cr.scalebroad)
        out, st2 = ctx.rates4(temps, cr.scalebroad)
        ch, _ = ctx.rates4_channels(temps[:2], cr.scalebroad)
        nu, _ = ctx.rates4_nu(temps[:4], cr.scalebroad)
    assert st["accepted"] == st2["accepted"]
    for got, n in ((out, 8), (ch.sum(1), 2), (nu.sum(1), 4)):
        assert np.max(np.abs(got - ref[:n])[ref[:n] > 0] / ref[:n][ref[:n] > 0]) <= 1e-12
