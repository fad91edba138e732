"""The BPNN kernel's pair queues at their edges: atoms with no, one and two
neighbours, 32 and 33 and more than 64 pairs per lane, a list capacity above
256 (two-word queue entries), G4 only (pairs beyond R_c left out) against G4
with a G5 group (every pair), each against the oracle at the FP64 bars and
(mixed) the mixed bars of test_gpu_bpnn."""
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


def model(g5):
    m = W.maise_like_bpnn(0, rc=5.0)
    if g5:
        m.ang_kind = m.ang_kind.copy()
        m.ang_kind[-3:] = 5   # the last eta group's functions
    return m


def clusters():
    rng = np.random.default_rng(3)
    far = np.array([[0.0, 0, 0], [40, 0, 0], [42.5, 0, 0], [80, 0, 0], [82.5, 0, 0], [81, 2.2, 0]])
    ball = rng.normal(0, 1, (60, 3))
    ball *= (4.4 * rng.uniform(0, 1, (60, 1)) ** (1 / 3) / np.linalg.norm(ball, axis=1)[:, None])
    keep = [0]
    for i in range(60):   # no pair closer than 1.4 A
        if np.min(np.linalg.norm(ball[keep] - ball[i], axis=1)) > 1.4:
            keep.append(i)
    lat = W.fcc_lattice(3, 3, 3, 3.4) + rng.normal(0, 0.05, (108, 3))   # ~70 neighbours, periodic
    return [(far, 100.0, 0, 0), (ball[keep] + 15, 30.0, 0, 0), (np.mod(lat, 10.2), 10.2, 1, 0),
            (np.mod(lat, 10.2), 10.2, 1, 264)]


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("g5", [False, True])
@pytest.mark.parametrize("which", range(4))
def test_pairs_of_every_count(mdk, ora, which, g5, prec):
    x, L, per, nmax = clusters()[which]
    m = model(g5)
    n = x.shape[0]
    ctx = mdk.Context([0] * 3, [L] * 3, [per] * 3, np.full(n, W.MASS_AL), prec)
    ctx.set_potential_bpnn(m)
    ctx.plan(m.rc, 0.3, nmax)
    ctx.set_state(x)
    E, F, Wv = ctx.compute()
    ref = ora.bpnn(x, [0] * 3, [L] * 3, [per] * 3, m)
    if prec == "fp64":
        assert abs(E[0] - ref["E"]) <= 1e-12 * abs(ref["E"])
        assert np.max(np.abs(F - ref["F"])) <= 1e-12 * np.max(np.abs(ref["F"])) + 1e-13
    else:
        assert abs(E[0] - ref["E"]) <= 2e-6 * n
        assert np.sqrt(np.mean((F - ref["F"]) ** 2)) <= 1e-4 * np.sqrt(np.mean(ref["F"] ** 2)) + 1e-12
    ctx.close()
