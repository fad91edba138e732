"""Kernels launched, as mdk_get_profile counts them, for runs whose launches can
be counted by hand: full LJ lists (one force kernel a step), one scan tile.  A
call of n steps runs the first kick, the check before the first step (one
kernel; 8 more where it builds), then as one loop the n - 1 plain steps: one
launch that sets their number, bodies of 8 force passes and a head, after a
body that builds or ends on the other gather copy 9 more; then the last force
pass."""
import numpy as np
import pytest

from paper_2511_22951_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def by_hand(n, every):
    since, total = 1, 1 + 1                 # kick, check
    if every and since >= every:
        total, since = total + 8, 0
    left = n - 1
    total += 1
    while left:
        e = min(8, left)
        if every:
            e = min(e, max(1, every - since))
        left, since, total = left - e, since + e, total + 9
        build = every and since >= every
        if build:
            since = 0
        if build or e % 2:
            total += 9
    return total + 1, since


@pytest.mark.parametrize("every", [0, 1, 3, 4, 11])
def test_counts(mdk, every):
    rng = np.random.default_rng(1)
    s = W.lattice_system(rng, (5, 5, 5), 5.26, W.MASS_AR, 20.0, sigma_jitter=0.02)
    ctx = mdk.Context(s.lo, s.hi, s.periodic, s.masses, "mixed")
    ctx.set_potential_lj(W.LJ_AR.eps, W.LJ_AR.sigma, W.LJ_AR.rc, 1)
    ctx.plan(W.LJ_AR.rc, 0.3, 0, every)
    ctx.set_launch(1, 128)
    ctx.set_state(s.x, s.v)
    for _ in range(4):                      # every graph captured
        ctx.step(0.01, 4)
    for n in (4, 8, 9, 10, 17, 18, 40, 41):
        ctx.build_neighbors(W.LJ_AR.rc, 0.3)   # since_build = 0
        ctx.step(0.01, 3)                       # forces valid again
        ctx.build_neighbors(W.LJ_AR.rc, 0.3)
        ctx.compute()
        ctx.profile(False)
        ctx.step(0.01, n)
        assert ctx.get_profile()["kernels"] == by_hand(n, every)[0], n
    ctx.close()
