"""When a step's rebuild chain runs as a graph: launched kernel by kernel the
first time it is met (a program that steps once captures nothing but the loop),
as a graph from the second time on, whatever dt is (a step size that changes
with every call, also under a thermostat, whose noise amplitudes follow it, and
with new knots).  Shown by the counted launches -- 1 for a chain in a graph that
does not build, 9 one by one -- and by the time of a call, which a new graph
would multiply (3 times the time at constant dt is the bar; capturing one takes
over 10 times that)."""
import time

import numpy as np
import pytest

from paper_2511_22951_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def context(mdk, lang):
    rng = np.random.default_rng(1)
    s = W.lattice_system(rng, (5, 5, 5), 5.26, W.MASS_AR, 20.0, sigma_jitter=0.02)
    ctx = mdk.Context(s.lo, s.hi, s.periodic, s.masses, "fp64")
    ctx.set_potential_lj(W.LJ_AR.eps, W.LJ_AR.sigma, W.LJ_AR.rc, 1)
    ctx.plan(W.LJ_AR.rc, 0.3)
    ctx.set_launch(1, 128)
    ctx.set_state(s.x, s.v)
    if lang:
        ctx.set_langevin([(-1e9, 1e9, 20.0, (0.0, 0.0, 0.0), 1e-4)], seed=5)
    ctx.compute()
    return ctx


def launches(ctx, dt, n):
    ctx.profile(False)
    ctx.step(dt, n)
    return ctx.get_profile()["kernels"]


@pytest.mark.parametrize("lang", [False, True])
def test_changing_dt(mdk, lang):
    ctx = context(mdk, lang)
    first = [launches(ctx, 0.01, 1) for _ in range(4)]
    assert first == [11, 11, 3, 3]          # kick, chain, force pass; one chain per gather copy
    assert [launches(ctx, 0.01 * (1.0 + 0.01 * k), 1) for k in range(6)] == [3] * 6

    def call_time(dts):
        t = []
        for dt in dts:
            a = time.perf_counter()
            ctx.step(dt, 1)
            t.append(time.perf_counter() - a)
        return np.median(t)

    call_time([0.01] * 20)
    same = call_time([0.01] * 40)
    assert call_time([0.01 * (1.5 + 0.01 * k) for k in range(40)]) < 3.0 * same
    ctx.close()


def test_first_call_captures_the_loop_only(mdk):
    ctx = context(mdk, False)
    # kick 1, chain one by one 9, set 1, body 9, last force pass 1
    assert launches(ctx, 0.001, 9) == 21
    ctx.close()
