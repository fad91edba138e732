"""Which of its two atoms' lists keeps a pair: every atom of an fcc lattice
keeps exactly half of its neighbours (each vector d has its opposite, and no
lattice vector in reach is level along the rule's direction); atoms at the
same place, images of an atom itself and lists filtered from an outer list
still hold one of each mirror pair."""
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
    i = np.repeat(np.arange(n, dtype=np.int64), np.diff(off))
    c = (im[:, 0].astype(np.int64) + 1) + 3 * (im[:, 1] + 1) + 9 * (im[:, 2] + 1)
    return np.sort((i * n + j) * 27 + c)


def lists(mdk, x, L, rc, outer=None):
    n, out = len(x), []
    for kind in ("full", "half"):
        ctx = mdk.Context(np.zeros(3), L, (1, 1, 1), np.full(n, W.MASS_AR), "fp64")
        ctx.set_potential_lj(W.LJ_AR.eps, 2.0, rc, 1)
        ctx.plan(rc, 0.3)
        if outer:
            ctx.set_outer_skin(outer)
        ctx.set_list_kind(kind)
        ctx.set_state(x)
        ctx.build_neighbors(rc, 0.3)
        out.append(ctx.neighbors())
        ctx.close()
    return out


@pytest.mark.parametrize("cells", [3, 4, 6])     # 2, 2 and 3 grid cells a side
def test_fcc_atoms_keep_half(mdk, cells):
    a = 5.26
    base = np.array([[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0]])
    g = np.stack(np.meshgrid(*[np.arange(cells)] * 3, indexing="ij"), -1).reshape(-1, 1, 3)
    x = (g + base).reshape(-1, 3) * a + 0.1
    full, half = lists(mdk, x, np.full(3, cells * a), 8.5 if cells > 3 else 7.0)
    assert np.array_equal(2 * np.diff(half[0]), np.diff(full[0]))


@pytest.mark.parametrize("outer", [None, 1.5])
def test_one_of_each_mirror_pair(mdk, outer):
    rng = np.random.default_rng(5)
    L = np.array([14.5, 15.0, 22.0])
    x = np.repeat(rng.uniform(0, 1, (150, 3)) * L, 2, axis=0)     # pairs at one place
    n = len(x)
    full, half = (keys(n, *q) for q in lists(mdk, x, L, 5.0, outer))
    c, ij = half % 27, half // 27
    both = np.concatenate([half, ((ij % n) * n + ij // n) * 27 + (26 - c)])
    assert np.array_equal(np.sort(both), full)
