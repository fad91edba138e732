"""Candidates outside the reach of a slice's bounding box are left out before
the pair tests: pairs at exactly the list radius along the box's axes, slices
whose box is a point or a small clump in a wide cell, more than one tile of
candidates of which most are out of reach, and a slice with a far atom (no
box).  Lists are integers: they equal the oracle's."""
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


def lattice():          # spacing 2.9: pairs at exactly rc + skin = 5.8, atoms on cell faces
    g = np.arange(8) * 2.9
    return np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3), (23.2,) * 3, (1, 1, 1)


def clumps():           # cells of 8.6 (radius 5.8), clumps of 40 within 0.6 of one point each
    rng = np.random.default_rng(1)
    c = rng.uniform(0, 1, (64, 3)) * 25.8
    x = (c[:, None, :] + rng.uniform(0, 0.6, (64, 40, 3))).reshape(-1, 3) % 25.8
    return x, (25.8,) * 3, (1, 1, 1)


def lone():             # one atom per occupied cell at most times: a box of one point
    rng = np.random.default_rng(2)
    return rng.uniform(0, 1, (300, 3)) * 100.0, (100.0,) * 3, (1, 0, 1)


def far():              # atoms far outside a free box share end cells with near ones
    rng = np.random.default_rng(3)
    x = rng.uniform(0, 1, (900, 3)) * 20.0
    x[::9] += rng.normal(0, 300.0, (100, 3))
    return x, (20.0,) * 3, (0, 0, 0)


@pytest.mark.parametrize("kind", ["full", "half"])
@pytest.mark.parametrize("make", [lattice, clumps, lone, far])
def test_lists_equal_the_oracle(mdk, ora, make, kind):
    x, L, per = make()
    n, L = len(x), np.array(L)
    rc, skin = 5.5, 0.3
    ctx = mdk.Context(np.zeros(3), L, per, np.full(n, W.MASS_AR), "mixed")
    ctx.set_potential_lj(W.LJ_AR.eps, 2.0, rc, 1)
    ctx.plan(rc, skin)
    ctx.set_list_kind(kind)
    ctx.set_state(x)
    ctx.build_neighbors(rc, skin)
    got = keys(n, *ctx.neighbors())
    ref = ora.neighbors(x, np.zeros(3), L, per, rc + skin, method="brute")
    rows = np.concatenate(ref)
    want = keys(n, np.concatenate([[0], np.cumsum([q.shape[0] for q in ref])]), rows[:, 0], rows[:, 1:])
    if kind == "half":
        c, ij = got % 27, got // 27
        got = np.sort(np.concatenate([got, ((ij % n) * n + ij // n) * 27 + (26 - c)]))
    assert np.array_equal(got, want)
    ctx.close()
