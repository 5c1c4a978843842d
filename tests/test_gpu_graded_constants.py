"""Force constants whose blocks differ by many orders of magnitude between sublattices, with modes that live on one
sublattice each: the ++ and -- parts of such a crystal come from vertices 1e-8 times the largest of their block, and have
to reach the FP64 bar like the others (a contraction in fixed point below one scale per block would lose them); a list
whose small quartets are not symmetric in their legs has to be evaluated as it is given."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2104_04895_gb300 import synth
from paper_2104_04895_gb300.binding import FP_OK, FP_PREC_DOUBLE_FLOAT, FP_PREC_FP64, Context, fp_stats

from conftest import oracle_modes

pytestmark = pytest.mark.gpu

RTOL = 1e-10  # the FP64 bar of the library
WEAK = 1e-8


def _crystal(maker, light):
    """Quartets with three or four legs on the atoms `light` scaled by WEAK."""
    cr = maker()
    n = np.isin(cr.fc4_idx[:, :4], light).sum(1)
    cr.fc4_val = cr.fc4_val * np.where(n >= 3, WEAK, 1.0)[:, None]
    return cr, n >= 3


def _modes(cr, light, seed):
    """Half of the branches on the atoms `light` at 10 rad/ps, the others on the rest at 30: 30 = 10 + 10 + 10 are the
    only ++ and -- processes.  Exact time reversal."""
    rng = np.random.Generator(np.random.PCG64(seed))
    N, nb = cr.nq, cr.nb
    G = np.stack(np.unravel_index(np.arange(N), cr.grid), 1)
    neg = np.ravel_multi_index(tuple(((-G) % np.array(cr.grid)).T), cr.grid)
    comp = [np.array([3 * a + c for a in atoms for c in range(3)])
            for atoms in (light, [a for a in range(cr.natoms) if a not in light])]
    h = nb // 2
    assert len(comp[0]) == h
    w, e, v = np.zeros((N, nb)), np.zeros((N, nb, nb), complex), np.zeros((N, nb, 3))
    for q in range(N):
        p = neg[q]
        if p < q:
            w[q], e[q], v[q] = w[p], e[p].conj(), -v[p]
            continue
        for s in range(2):
            m = rng.normal(size=(h, h)) + (1j * rng.normal(size=(h, h)) if p != q else 0.0)
            u = np.linalg.qr(m)[0]
            e[q][np.ix_(np.arange(s * h, (s + 1) * h), comp[s])] = u
            w[q, s * h:(s + 1) * h] = np.sort(rng.uniform(9.7, 10.3, h) * (1.0, 3.0)[s])
        v[q] = rng.normal(size=(nb, 3)) if p != q else 0.0
    return w, e, v


CASES = [(lambda: synth.zincblende_bas((3, 2, 2)), [1]), (lambda: synth.licoo2((3, 1, 1)), [2, 3])]


def _close(got, ref):
    assert (ref > 0).any()
    zero = ref == 0.0
    assert np.all(got[zero] == 0.0)
    assert np.max(np.abs(got[~zero] - ref[~zero]) / ref[~zero]) <= RTOL


@pytest.mark.parametrize("precision", [FP_PREC_FP64, FP_PREC_DOUBLE_FLOAT])
@pytest.mark.parametrize("temps", [[300.0], [250.0, 900.0]])
@pytest.mark.parametrize("maker,light", CASES)
def test_weak_vertices_keep_their_accuracy(maker, light, temps, precision):
    cr, _ = _crystal(maker, light)
    w, e, v = _modes(cr, light, 3)
    nT = len(temps)
    refs = [oracle.rates4(cr, w, e, v, temps=temps, processes=(p,)) for p in range(3)]
    full, acc = oracle.rates4(cr, w, e, v, temps=temps)
    with Context.from_crystal(cr) as ctx:
        ctx.set_modes(w, e, v)
        ch, st = ctx.rates4_channels(temps, cr.scalebroad, precision=precision)
        assert st["accepted"] == [refs[p][1][p] for p in range(3)]
        for p in range(3):
            _close(ch[:, p].reshape(nT, -1), refs[p][0])
            one, _ = ctx.rates4(temps, cr.scalebroad, precision=precision, process_mask=1 << p)
            _close(one.reshape(nT, -1), refs[p][0])
        out, st = ctx.rates4(temps, cr.scalebroad, precision=precision)
        _close(out.reshape(nT, -1), full)
        assert st["accepted"] == list(acc)


@pytest.mark.parametrize("maker,light", CASES)
def test_weak_vertices_without_allocation(maker, light):
    import torch
    cr, _ = _crystal(maker, light)
    w, e, v = _modes(cr, light, 5)
    T = np.array([300.0])
    ref, acc = oracle.rates4(cr, w, e, v, temps=T, processes=(2,))
    with Context.from_crystal(cr) as ctx:
        ctx.set_modes(w, e, v)
        out = torch.zeros(cr.nq * cr.nb, dtype=torch.float64, device="cuda")
        o, st = ctx.make_opts(process_mask=4)[0], fp_stats()
        rc = ctx.L.fp_rates4_noalloc(ctx.h, 1, T.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), cr.scalebroad,
                                     ctypes.byref(o), ctypes.c_void_p(out.data_ptr()), ctypes.byref(st))
        assert rc == FP_OK, ctx.L.fp_last_error(ctx.h)
        _close(out.cpu().numpy().reshape(1, -1), ref)
        assert list(st.accepted) == list(acc)


@pytest.mark.parametrize("maker,light", CASES)
def test_small_asymmetric_quartets_count(maker, light):
    """The small quartets lose the symmetry under i <-> j by 1e-5 of their size (1e-13 of the largest quartet), keeping
    that under j <-> k, which every path needs."""
    cr, small = _crystal(maker, light)
    w, e, v = _modes(cr, light, 4)
    rng = np.random.Generator(np.random.PCG64(6))
    n = len(cr.fc4_idx)
    d = rng.normal(0.0, 1e-5 * WEAK, cr.fc4_val.shape) * small[:, None]
    order = {tuple(k): i for i, k in enumerate(cr.fc4_idx)}
    perm = np.array([order[tuple(k)] for k in cr.fc4_idx[:, [0, 2, 1, 3, 7, 8, 9, 4, 5, 6, 10, 11, 12]]])
    cr.fc4_val = cr.fc4_val + 0.5 * (d + d[perm].reshape(n, 3, 3, 3, 3).transpose(0, 1, 3, 2, 4).reshape(n, 81))
    with Context.from_crystal(cr) as ctx:
        ctx.set_modes(w, e, v)
        for p in (0, 2):
            ref, _ = oracle.rates4(cr, w, e, v, processes=(p,))
            out, _ = ctx.rates4(cr.temps, cr.scalebroad, process_mask=1 << p)
            _close(out.reshape(len(cr.temps), -1), ref)


@pytest.mark.parametrize("maker", [lambda: synth.diamond_si((4, 3, 3)), lambda: synth.zincblende_bas((4, 3, 2)),
                                   lambda: synth.licoo2((3, 2, 2))])
@pytest.mark.parametrize("temps", [[300.0], [20.0, 100.0, 900.0]])
def test_ordinary_crystals_keep_the_fast_contraction(maker, temps):
    """Every entry of an evaluated row is formed there, exactly one per accepted term in the other pair kernels."""
    cr = maker()
    w, e, v = oracle_modes(cr)
    with Context.from_crystal(cr) as ctx:
        ctx.set_modes(w, e, v)
        _, st = ctx.rates4(temps, cr.scalebroad)
        assert st["vertex_entries"] != st["terms_executed"]
