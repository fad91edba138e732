"""The list build's slices and tiles at their edges: systems on every slice
length (8, 16 and 32 atoms), cells whose template holds more candidates than
one tile (1024), single-atom and empty cells, and free boxes whose atoms lie
outside (clamped into end cells, beyond 0.6 and 2 cell sizes).  Lists are
integers, so they equal the oracle's exactly; the half list holds one of each
mirror pair."""
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


def keys(n, off, j, im):
    """One sorted integer per entry (i, j, image)."""
    i = np.repeat(np.arange(n, dtype=np.int64), np.diff(off))
    c = (im[:, 0].astype(np.int64) + 1) + 3 * (im[:, 1] + 1) + 9 * (im[:, 2] + 1)
    return np.sort((i * n + j) * 27 + c)


def mirrored(n, k):
    c, ij = k % 27, k // 27
    return np.sort(((ij % n) * n + ij // n) * 27 + (26 - c))


#        atoms  box lengths            periodic   spread
CASES = [
    (1, (20.0, 20.0, 20.0), (1, 1, 1), "uniform"),
    (700, (60.0, 55.0, 50.0), (1, 1, 1), "uniform"),      # cells of 0 to 5 atoms
    (1750, (18.0, 18.5, 18.9), (1, 1, 1), "uniform"),     # ~64 per cell: two tiles, self images
    (400, (20.0, 20.0, 20.0), (0, 0, 0), "cluster"),      # most atoms outside the box
    (16384, (70.0, 60.0, 50.0), (1, 1, 0), "uniform"),    # slices of 16
    (66000, (60.0, 60.0, 60.0), (1, 1, 1), "uniform"),    # slices of 32, ~66 per cell: two tiles
]


@pytest.mark.parametrize("case", CASES)
def test_lists_equal_the_oracle(mdk, ora, case):
    n, L, per, spread = case
    rc, skin = 5.5, 0.3
    rng = np.random.default_rng(n)
    L = np.array(L)
    x = rng.uniform(0, 1, (n, 3)) * L if spread == "uniform" else 10.0 + rng.normal(0, 14.0, (n, 3))
    ctx = mdk.Context(np.zeros(3), L, per, np.full(n, W.MASS_AR), "mixed")
    ctx.set_potential_lj(W.LJ_AR.eps, 2.0, rc, 1)
    ctx.plan(rc, skin)
    ctx.set_state(x)
    ctx.build_neighbors(rc, skin)
    full = keys(n, *ctx.neighbors())
    ref = ora.neighbors(x, np.zeros(3), L, per, rc + skin, method="brute" if n < 2000 else "cells")
    off = np.concatenate([[0], np.cumsum([q.shape[0] for q in ref])])
    rows = np.concatenate(ref)
    assert np.array_equal(full, keys(n, off, rows[:, 0], rows[:, 1:]))
    ctx.set_list_kind("half")
    ctx.build_neighbors(rc, skin)
    half = keys(n, *ctx.neighbors())
    assert 2 * half.size == full.size
    assert np.array_equal(np.sort(np.concatenate([half, mirrored(n, half)])), full)
    ctx.close()
