"""Behler-Parrinello models with G5 functions take the kernel instance of their
own group count: parity with the oracle for 1 to 8 (eta, kind) groups, G5 only
and G4 / G5 mixed, below and above 32 neighbours (the two gradient schedules);
and the list capacity that a model leaves room for: 227 KB of shared memory
hold the weights and, for the one warp of the smallest launch, 14 reals, one
per compiled group and an int per list slot.  Bars as in test_gpu_bpnn."""
import numpy as np
import pytest

from paper_2511_22951_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def model(groups, kinds, rc=5.0):
    """groups (eta, kind) groups of 8 functions; kinds: 5, 4 or 45 (in turn)."""
    m = W.maise_like_bpnn(0, rc=rc, n_ang=8)
    z, lam = m.ang_par[:, 0], m.ang_par[:, 1]
    etas = np.geomspace(0.0005, 0.06, groups)
    m.ang_par = np.concatenate([np.stack([z, lam, np.full(8, e)], 1) for e in etas])
    k = [5 if kinds == 5 or (kinds == 45 and g % 2 == 0) else 4 for g in range(groups)]
    m.ang_kind = np.repeat(np.array(k, dtype=np.int32), 8)
    rng = np.random.default_rng(9)
    m.W01 = rng.normal(0.0, 0.05, size=(8 + 8 * groups, 10))
    return m


def check(mdk, ora, m, x, L, prec, nmax=0):
    n = x.shape[0]
    ctx = mdk.Context([0] * 3, [L] * 3, [1] * 3, np.full(n, W.MASS_AL), prec)
    ctx.set_potential_bpnn(m)
    ctx.plan(m.rc, 0.3, nmax)
    ctx.set_state(x)
    E, F, _ = ctx.compute()
    ctx.close()
    ref = ora.bpnn(x, [0] * 3, [L] * 3, [1] * 3, m)
    if prec == "fp64":
        assert abs(E[0] - ref["E"]) <= 1e-12 * abs(ref["E"])
        assert np.max(np.abs(F - ref["F"])) <= 1e-12 * np.max(np.abs(ref["F"])) + 1e-13
    else:
        assert abs(E[0] - ref["E"]) <= 2e-6 * n
        assert np.sqrt(np.mean((F - ref["F"]) ** 2)) <= 1e-4 * np.sqrt(np.mean(ref["F"] ** 2)) + 1e-12


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("a", [5.2, 3.6])         # 18 and 54 neighbours within R_c
@pytest.mark.parametrize("groups,kinds", [(1, 5), (2, 45), (3, 5), (4, 45), (5, 45), (6, 5), (8, 45)])
def test_every_group_count(mdk, ora, groups, kinds, a, prec):
    rng = np.random.default_rng(groups)
    x = W.fcc_lattice(3, 3, 3, a) + rng.normal(0, 0.05, (108, 3))
    check(mdk, ora, model(groups, kinds), np.mod(x, 3 * a), 3 * a, prec)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("kinds", [4, 45])
def test_more_neighbours_than_a_round_packs(mdk, ora, kinds, prec):
    """~226 neighbours: past the 192 that a mixed round packs at a time.  Input
    weights down by the pair count (226^2 / 54^2), so that the first layer is
    not saturated (its reverse pass takes 1 - h^2)."""
    rng = np.random.default_rng(4)
    x = W.fcc_lattice(4, 4, 4, 2.1) + rng.normal(0, 0.03, (256, 3))
    m = model(2, kinds)
    m.W01 = m.W01 * (54.0 / 226.0) ** 2
    check(mdk, ora, m, np.mod(x, 8.4), 8.4, prec)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("groups,kinds", [(2, 5), (6, 45), (2, 4), (6, 4)])
def test_list_capacity(mdk, ora, groups, kinds, prec):
    r = 8 if prec == "fp64" else 4
    weights = (72 * 10 + 10 + 10 * 10 + 20) * r
    fixed = (2 * 80 + 96 + 64) * r
    nmax = (227 * 1024 - (weights + 15) // 16 * 16 - fixed - 16) // ((14 + groups) * r + 4) // 8 * 8
    rng = np.random.default_rng(3)
    x = W.fcc_lattice(3, 3, 3, 3.6) + rng.normal(0, 0.05, (108, 3))
    check(mdk, ora, model(groups, kinds), np.mod(x, 10.8), 10.8, prec, nmax)
