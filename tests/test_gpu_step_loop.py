"""Captured step loops against eager steps: runs of every length around a loop
body (8 places), odd ends, triggers at any place, fixed build intervals that
cut a body, thermo samples that cut a run, two-level lists (whose filter
builds leave the gather copy alone) and Langevin noise (keyed by the step
index).  The same kernels run in the same order, so positions, velocities,
samples and build counts are bitwise those of eager steps."""
import numpy as np
import pytest

from paper_2511_22951_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mdk():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_22951_gb300 import _build, mdk as m
    _build.build()
    m.load()
    return m


def run(mdk, graphs, runs, every, thermo, outer, lang, prec):
    rng = np.random.default_rng(11)
    s = W.lattice_system(rng, (5, 5, 6), 5.3, W.MASS_AR, 400.0, sigma_jitter=0.1)
    ctx = mdk.Context(s.lo, s.hi, s.periodic, s.masses, prec)
    ctx.set_potential_lj(W.LJ_AR.eps, W.LJ_AR.sigma, W.LJ_AR.rc, 1)
    ctx.plan(W.LJ_AR.rc, 0.3, 0, every)
    if outer:
        ctx.set_outer_skin(1.5)
    if thermo:
        ctx.set_thermo(thermo, 64)
    ctx.set_graphs(graphs)
    ctx.set_launch(1, 128)
    if lang:
        ctx.set_langevin([(-1e9, 1e9, 400.0, (0.0, 0.0, 0.0), 0.01)], seed=5)
    ctx.set_state(s.x, s.v)
    for n in runs:
        ctx.step(3.0, n)
    x, v = ctx.get_state()
    t = ctx.thermo() if thermo else np.zeros(0)
    c = ctx.counters(), ctx.build_counts()
    ctx.close()
    return x, v, t, c


@pytest.mark.parametrize("runs,every,thermo,outer,lang,prec", [
    ((1, 2, 3, 4, 5, 6, 7), 0, 0, 0, 0, "mixed"),
    ((8, 9, 10, 11, 17, 18, 19, 40), 0, 0, 0, 0, "fp64"),
    ((30, 31), 1, 0, 0, 0, "mixed"),
    ((30, 31), 3, 0, 0, 1, "mixed"),
    ((41,), 5, 0, 1, 0, "mixed"),
    ((60, 37), 0, 0, 1, 1, "mixed"),
    ((60, 37), 0, 7, 1, 0, "fp64"),
    ((50,), 4, 10, 0, 0, "mixed"),
])
def test_loop_equals_eager(mdk, runs, every, thermo, outer, lang, prec):
    a = run(mdk, True, runs, every, thermo, outer, lang, prec)
    b = run(mdk, False, runs, every, thermo, outer, lang, prec)
    assert a[3] == b[3]
    assert a[3][0][1] == sum(runs)
    for p, q in zip(a[:3], b[:3]):
        assert np.array_equal(p, q)
