"""The pair kernel (FP64 and double-float paths on force constants with the transposition symmetry of Eq. TS) at the
places where its bookkeeping can go wrong: points that are their own -q beside real pairs, masks that select only one
member or some branches of a pair, branch chunks of one pair, several temperatures, single processes, the form
without a slot per pair, and force constants without the symmetry (which take the other kernel)."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2104_04895_gb300 import synth
from paper_2104_04895_gb300.binding import FP_OK, FP_PREC_DOUBLE_FLOAT, FP_PREC_FP64, Context, fp_stats

from conftest import oracle_modes

pytestmark = pytest.mark.gpu

RTOL = 1e-10  # the FP64 bar of the library


def _close(got, ref):
    zero = ref == 0.0
    assert np.all(got[zero] == 0.0)
    assert np.max(np.abs(got[~zero] - ref[~zero]) / np.abs(ref[~zero]), initial=0.0) <= RTOL


@pytest.mark.parametrize("precision", [FP_PREC_FP64, FP_PREC_DOUBLE_FLOAT])
@pytest.mark.parametrize("maker,temps,opts", [
    (lambda: synth.simple_cubic((4, 3, 1)), [300.0], {}),
    (lambda: synth.simple_cubic((5, 2, 2)), [300.0, 500.0, 900.0], dict(block_j0=1)),
    (lambda: synth.diamond_si((2, 3, 2)), [300.0], dict(block_j0=2, threads=96)),
    (lambda: synth.zincblende_bas((3, 2, 2)), list(np.linspace(250.0, 950.0, 8)), {}),
    (lambda: synth.zincblende_bas((3, 2, 2)), [400.0], dict(no_time_reversal=1, k1_tile=5)),
    (lambda: synth.licoo2((2, 1, 2)), [300.0], {}),
    (lambda: synth.licoo2((3, 1, 1)), [300.0, 600.0], dict(block_j0=1)),
])
def test_masks_chunks_and_processes(precision, maker, temps, opts):
    cr = maker()
    w, e, v = oracle_modes(cr)
    N, nb, nT = cr.nq, cr.nb, len(temps)
    rng = np.random.Generator(np.random.PCG64(N * nb + nT))
    with Context.from_crystal(cr) as ctx:
        ctx.set_modes(w, e, v)
        for mask in (None, (rng.random(N * nb) < 0.4).astype(np.uint8)):
            sel = np.arange(N * nb) if mask is None else np.nonzero(mask)[0]
            ref, acc = oracle.rates4(cr, w, e, v, temps=temps, sel=sel)
            out, st = ctx.rates4(temps, cr.scalebroad, precision=precision, mode_mask=mask, **opts)
            flat = out.reshape(nT, -1)
            _close(flat[:, sel], ref)
            assert np.all(np.delete(flat, sel, axis=1) == 0.0)
            assert st["accepted"] == list(acc)
            again, _ = ctx.rates4(temps, cr.scalebroad, precision=precision, mode_mask=mask, **opts)
            assert np.array_equal(out, again)
        for p in range(3):
            ref, acc = oracle.rates4(cr, w, e, v, temps=temps, processes=(p,))
            out, st = ctx.rates4(temps, cr.scalebroad, precision=precision, process_mask=1 << p, **opts)
            _close(out.reshape(nT, -1), ref)
            assert st["accepted"][p] == acc[p]


@pytest.mark.parametrize("precision", [FP_PREC_FP64, FP_PREC_DOUBLE_FLOAT])
def test_without_a_slot_per_pair(precision):
    """fp_rates4_noalloc where a slot per (point, q') exceeds its 16 MiB: every q' is evaluated, same rates."""
    import torch
    cr = synth.licoo2((5, 4, 3))
    temps = np.linspace(300.0, 1000.0, 8)
    with Context.from_crystal(cr) as ctx:
        ctx.modes(copy=False)
        mask = np.zeros((cr.nq, cr.nb), np.uint8)
        mask[1::7] = 1
        o, keep = ctx.make_opts(precision=precision, block_j0=1, mode_mask=mask.reshape(-1))
        ref, st = ctx.rates4(temps, cr.scalebroad, precision=precision, block_j0=1, mode_mask=mask.reshape(-1))
        full, st_full = ctx.make_opts(precision=precision, block_j0=1)[0], fp_stats()
        out = torch.zeros(len(temps) * cr.nq * cr.nb, dtype=torch.float64, device="cuda")
        T = np.ascontiguousarray(temps)
        for opt, s in ((o, fp_stats()), (full, st_full)):
            rc = ctx.L.fp_rates4_noalloc(ctx.h, len(T), T.ctypes.data_as(ctypes.POINTER(ctypes.c_double)),
                                         cr.scalebroad, ctypes.byref(opt), ctypes.c_void_p(out.data_ptr()),
                                         ctypes.byref(s))
            assert rc == FP_OK, ctx.L.fp_last_error(ctx.h)
            got = out.cpu().numpy().reshape(ref.shape)
            pick = mask.astype(bool)
            _close(got[:, pick], ref[:, pick])
        whole, st_w = ctx.rates4(temps, cr.scalebroad, precision=precision)
        _close(got, whole)
        assert list(st_full.accepted) == st_w["accepted"]
        del keep


@pytest.mark.parametrize("precision", [FP_PREC_FP64, FP_PREC_DOUBLE_FLOAT])
def test_force_constants_without_the_symmetry(precision):
    """Phi4 symmetric only under the exchange of legs j and k takes the kernel that uses no other exchange."""
    cr = synth.diamond_si((3, 2, 2))
    rng = np.random.Generator(np.random.PCG64(5))
    n = len(cr.fc4_idx)
    val = cr.fc4_val + rng.normal(0.0, 1.0, cr.fc4_val.shape)
    swapped = cr.fc4_idx[:, [0, 2, 1, 3, 7, 8, 9, 4, 5, 6, 10, 11, 12]]
    order = {tuple(k): i for i, k in enumerate(cr.fc4_idx)}
    perm = np.array([order[tuple(k)] for k in swapped])
    other = val[perm].reshape(n, 3, 3, 3, 3).transpose(0, 1, 3, 2, 4).reshape(n, 81)
    cr.fc4_val = 0.5 * (val + other)
    w, e, v = oracle_modes(cr)
    ref, acc = oracle.rates4(cr, w, e, v)
    with Context.from_crystal(cr) as ctx:
        ctx.set_modes(w, e, v)
        out, st = ctx.rates4(cr.temps, cr.scalebroad, precision=precision)
    _close(out.reshape(1, -1), ref)
    assert st["accepted"] == list(acc)


@pytest.mark.parametrize("precision", [FP_PREC_FP64, FP_PREC_DOUBLE_FLOAT])
@pytest.mark.parametrize("maker", [lambda: synth.diamond_si((3, 2, 2)), lambda: synth.licoo2((2, 1, 2))])
def test_eigenvectors_of_any_norm(precision, maker):
    """Mode tables whose eigenvectors are not of unit norm take the contraction that has no fixed-point scale."""
    cr = maker()
    w, e, v = oracle_modes(cr)
    f = 2.0 ** np.arange(cr.nb) * 1.1  # the same at q and -q
    e = e * f[None, :, None]
    ref, acc = oracle.rates4(cr, w, e, v)
    with Context.from_crystal(cr) as ctx:
        ctx.set_modes(w, e, v)
        out, st = ctx.rates4(cr.temps, cr.scalebroad, precision=precision)
    _close(out.reshape(len(cr.temps), -1), ref)
    assert st["accepted"] == list(acc)


@pytest.mark.parametrize("scale", [1e-90, 1e-30, 3.0, 1e60])
def test_force_constants_of_any_size(scale):
    """The fixed-point scale of the contraction follows Phi4: the rates scale with its square."""
    cr = synth.zincblende_bas((3, 2, 2))
    w, e, v = oracle_modes(cr)
    ref, _ = oracle.rates4(cr, w, e, v)
    with Context.from_crystal(cr.scaled_fc4(scale)) as ctx:
        ctx.set_modes(w, e, v)
        out, _ = ctx.rates4(cr.temps, cr.scalebroad)
    _close(out.reshape(1, -1) / scale ** 2, ref)


def _close_parts(got, ref):
    """_close where a part of a symmetric grid may hold only vertices that vanish: rounding, 1e-30 of the others, on both
    sides."""
    noise = np.abs(ref) <= 1e-20 * ref.max()
    assert np.all(np.abs(got[noise]) <= 1e-20 * ref.max())
    _close(got[~noise], ref[~noise])


@pytest.mark.parametrize("precision", [FP_PREC_FP64, FP_PREC_DOUBLE_FLOAT])
@pytest.mark.parametrize("maker,nT", [(lambda: synth.simple_cubic((4, 3, 2)), 1), (lambda: synth.zincblende_bas((3, 2, 2)), 2),
                                      (lambda: synth.licoo2((2, 1, 2)), 4), (lambda: synth.diamond_si((2, 2, 2)), 5)])
def test_parts_in_one_pass(precision, maker, nT):
    """Normal and Umklapp parts and the channels: one pass up to eight sums per mode (2 nT, 3 nT), passes beyond."""
    cr = maker()
    w, e, v = oracle_modes(cr)
    temps = list(np.linspace(300.0, 900.0, nT))
    N, nb = cr.nq, cr.nb
    rng = np.random.Generator(np.random.PCG64(N))
    mask = (rng.random(N * nb) < 0.5).astype(np.uint8)
    with Context.from_crystal(cr) as ctx:
        ctx.set_modes(w, e, v)
        nu, st = ctx.rates4_nu(temps, cr.scalebroad, precision=precision)
        nm, st_m = ctx.rates4_nu(temps, cr.scalebroad, precision=precision, mode_mask=mask, process_mask=6)
        ch, st_c = ctx.rates4_channels(temps, cr.scalebroad, precision=precision)
        full, st_f = ctx.rates4(temps, cr.scalebroad, precision=precision)
    total = np.zeros(3)
    for p, name in enumerate(("normal", "umklapp")):
        ref, acc = oracle.rates4(cr, w, e, v, temps=temps, nu=name)
        _close_parts(nu[:, p].reshape(nT, -1), ref)
        total += acc
        sel = np.nonzero(mask)[0]
        ref, _ = oracle.rates4(cr, w, e, v, temps=temps, nu=name, sel=sel, processes=(1, 2))
        _close_parts(nm[:, p].reshape(nT, -1)[:, sel], ref)
        assert np.all(nm[:, p].reshape(nT, -1)[:, mask == 0] == 0.0)
    for p in range(3):
        ref, acc = oracle.rates4(cr, w, e, v, temps=temps, processes=(p,))
        _close_parts(ch[:, p].reshape(nT, -1), ref)
        assert st_c["accepted"][p] == acc[p]
    assert st["accepted"] == list(total) == st_f["accepted"]
    assert st["candidates"] == 2 * st_f["candidates"] and st_c["candidates"] == st_f["candidates"]


@pytest.mark.parametrize("precision", [FP_PREC_FP64, FP_PREC_DOUBLE_FLOAT])
@pytest.mark.parametrize("maker,nT", [(lambda: synth.simple_cubic((2, 1, 2)), 1), (lambda: synth.simple_cubic((4, 3, 3)), 1),
                                      (lambda: synth.diamond_si((2, 2, 1)), 3), (lambda: synth.diamond_si((4, 3, 3)), 1)])
def test_several_items_per_pair(precision, maker, nT):
    """Grids whose pairs are dealt to several items (up to one per q'', and two of nine q'' each): rates, accepted counts and
    the per-mode counts of the phase space, which share the items' slots; block_j0 = 1 adds chunks to the slots."""
    cr = maker()
    w, e, v = oracle_modes(cr)
    temps = list(np.linspace(300.0, 900.0, nT))
    N, nb = cr.nq, cr.nb
    ref, acc = oracle.rates4(cr, w, e, v, temps=temps)
    ps, pacc = oracle.rates4(cr, w, e, v, temps=temps, unit_vertex=True)
    with Context.from_crystal(cr) as ctx:
        ctx.set_modes(w, e, v)
        for opts in ({}, dict(block_j0=1), dict(no_time_reversal=1)):
            out, st = ctx.rates4(temps, cr.scalebroad, precision=precision, **opts)
            _close_parts(out.reshape(nT, -1), ref)
            assert st["accepted"] == list(acc)
            npr, _, wp4 = ctx.phase_space4(temps, cr.scalebroad, precision=precision, **opts)
            _close(wp4.reshape(nT, -1) * N ** 2, ps)
            assert npr.sum() == pacc.sum()
