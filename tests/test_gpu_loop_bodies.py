"""Captured step loops against eager steps, bitwise, for what a loop body holds:
several kernels per place (EAM and half lists), forces straight from the cells,
BPNN, a piston, list builds that overflow inside a body, and bodies of 2 places
(large grids), whose odd end is a trigger at their first place.  Runs are odd
and even and cut by fixed build intervals.  FP64 half lists sum in any order:
there the two runs agree to rounding (1e-9 of the spread after these steps; one
step misplaced shows at 1e-3) and in their build counts."""
import numpy as np
import pytest

from paper_2511_22951_gb300 import workloads as W

pytestmark = pytest.mark.gpu


POTS = {  # potential: (lattice constant, mass, T, dt)
    "lj": (5.3, W.MASS_AR, 400.0, 3.0),
    "eam": (4.05, W.MASS_AL, 900.0, 2.0),
    "bpnn": (4.05, W.MASS_AL, 900.0, 2.0),
}


def run(mdk, graphs, pot, prec, kind, runs, every=0, outer=0.0, lang=False, cells=(5, 5, 6), tpa=1,
        piston=False, T=None, most=0):
    a, mass, T0, dt = POTS[pot]
    rng = np.random.default_rng(11)
    s = W.lattice_system(rng, cells, a, mass, T or T0, sigma_jitter=0.05)
    per, lo, hi = s.periodic, s.lo.copy(), s.hi.copy()
    if piston:
        per = [0, 1, 1]
        lo[0] -= 2 * a
        hi[0] += 8 * a
    ctx = mdk.Context(lo, hi, per, s.masses, prec)
    if pot == "lj":
        rc = W.LJ_AR.rc
        ctx.set_potential_lj(W.LJ_AR.eps, W.LJ_AR.sigma, rc, 1)
    elif pot == "eam":
        rc = W.AL_LIKE.rc
        ctx.set_potential_eam(W.tabulate_fs_eam(W.AL_LIKE))
    else:
        m = W.maise_like_bpnn(0, rc=5.0)
        rc = m.rc
        ctx.set_potential_bpnn(m)
    ctx.plan(rc, 0.3, most, every)
    if outer:
        ctx.set_outer_skin(outer)
    if kind != "full":
        ctx.set_list_kind(kind)
    ctx.set_launch(tpa, 128)
    ctx.set_graphs(graphs)
    ctx.set_state(s.x, s.v)
    ctx.build_neighbors(rc, 0.3)
    if piston:
        ctx.set_piston(0.02, (s.x[:, 0] < s.x[:, 0].min() + a).astype(np.uint8))
    if lang:
        ctx.set_langevin([(-1e9, 1e9, T or T0, (0.0, 0.0, 0.0), 0.01)], seed=5)
    for n in runs:
        ctx.step(dt, n)
    x, v = ctx.get_state()
    c = ctx.counters(), ctx.build_counts(), ctx.regrows
    ctx.close()
    return x, v, c


def check(mdk, exact=True, **k):
    a, b = run(mdk, True, **k), run(mdk, False, **k)
    assert a[2] == b[2] and a[2][0][1] == sum(k["runs"])
    for p, q in zip(a[:2], b[:2]):
        if exact:
            assert np.array_equal(p, q)
        else:
            assert np.max(np.abs(p - q)) <= 1e-9 * np.ptp(q)
    return a[2]


@pytest.mark.parametrize("runs,every", [((9, 10, 18, 31), 0), ((17, 12), 3), ((26, 11), 1)])
@pytest.mark.parametrize("pot,prec,kind", [
    ("eam", "mixed", "full"), ("eam", "fp64", "full"), ("eam", "mixed", "half"), ("lj", "mixed", "half"),
    ("lj", "fp64", "half"), ("eam", "fp64", "half"), ("lj", "mixed", "cells"), ("bpnn", "mixed", "full")])
def test_kernels_of_a_place(mdk, pot, prec, kind, runs, every):
    check(mdk, exact=not (prec == "fp64" and kind == "half"), pot=pot, prec=prec, kind=kind, runs=runs,
          every=every)


@pytest.mark.parametrize("pot,prec", [("lj", "mixed"), ("eam", "mixed"), ("lj", "fp64")])
def test_piston(mdk, pot, prec):
    check(mdk, pot=pot, prec=prec, kind="full", runs=(31, 10, 24), piston=True)


@pytest.mark.parametrize("prec,kind", [("mixed", "full"), ("fp64", "full"), ("mixed", "half")])
def test_overflow_inside_a_body(mdk, prec, kind):
    """Lists of 80 (half: 40) entries at most, outgrown as the crystal melts."""
    c = check(mdk, pot="lj", prec=prec, kind=kind, runs=(60, 21), T=3000.0,
              most=80 if kind == "full" else 40)
    assert c[2] >= 1


@pytest.mark.parametrize("runs,every,outer,lang", [
    ((2, 3, 4, 5), 0, 0.0, False), ((18, 7), 0, 0.0, True), ((11, 12), 3, 0.0, False),
    ((9, 8), 1, 0.0, False), ((21, 10), 0, 1.5, False), ((12, 9), 2, 1.5, True)])
def test_two_places(mdk, runs, every, outer, lang):
    """143,748 atoms, a warp per atom: 4.6 million lanes."""
    check(mdk, pot="lj", prec="mixed", kind="full", runs=runs, every=every, outer=outer, lang=lang,
          cells=(33, 33, 33), tpa=32)
