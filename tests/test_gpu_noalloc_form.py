"""fp_rates4_noalloc runs the kernel form that fp_rates4 runs wherever that fits its 16 MiB: the accepted terms a call
evaluated (one per unordered pair there, four times as many over ordered sums) and its vertex entries tell which ran."""
import ctypes

import numpy as np
import pytest

from paper_2104_04895_gb300 import synth
from paper_2104_04895_gb300.binding import FP_OK, FP_PREC_DOUBLE_FLOAT, FP_PREC_FP64, Context, fp_stats

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,maker,temps", [
    (FP_PREC_FP64, lambda: synth.diamond_si((8, 8, 8)), [300.0]),
    (FP_PREC_DOUBLE_FLOAT, lambda: synth.diamond_si((7, 7, 7)), [300.0]),
    (FP_PREC_FP64, lambda: synth.licoo2((5, 4, 3)), [300.0, 500.0, 700.0])])
def test_same_form_as_the_allocating_call(precision, maker, temps):
    import torch
    cr = maker()
    with Context.from_crystal(cr) as ctx:
        ctx.modes(copy=False)
        ref, st = ctx.rates4(temps, cr.scalebroad, precision=precision)
        T = np.ascontiguousarray(temps)
        out = torch.zeros(len(T) * cr.nq * cr.nb, dtype=torch.float64, device="cuda")
        o, got = ctx.make_opts(precision=precision)[0], fp_stats()
        rc = ctx.L.fp_rates4_noalloc(ctx.h, len(T), T.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), cr.scalebroad,
                                     ctypes.byref(o), ctypes.c_void_p(out.data_ptr()), ctypes.byref(got))
        assert rc == FP_OK, ctx.L.fp_last_error(ctx.h)
        assert got.terms_executed == st["terms_executed"] and got.vertex_entries == st["vertex_entries"]
        assert list(got.accepted) == st["accepted"]
        x = out.cpu().numpy().reshape(ref.shape)
        assert np.max(np.abs(x - ref)[ref > 0] / ref[ref > 0]) <= 1e-12
