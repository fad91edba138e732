"""The mixed full-list walks hand whole groups of 8 list entries to their
lanes: lane t of T takes groups t, t + T, ...  So where an atom's groups fit
the lanes of two launch shapes, each lane of both holds the same group and the
FP32 sums run in the same order: forces, energies, virials and the trajectory
are bitwise the same from T = (number of groups) lanes on, for LJ and EAM."""
import numpy as np
import pytest

from paper_2511_22951_gb300 import workloads as W

from test_gpu_parity import eam_ctx, lj_ctx

pytestmark = pytest.mark.gpu


# spacing over the cutoff, share of the sites taken, most entries: 12, 18 and
# 42 neighbours of the full lattice
LATTICES = [(1.35, 0.3, 8), (1.35, 1.0, 16), (0.95, 1.0, 32), (0.79, 1.0, 64)]


@pytest.mark.parametrize("pot", ["lj", "eam"])
@pytest.mark.parametrize("ratio,share,most", LATTICES)
def test_same_bits_from_enough_lanes(mdk, pot, ratio, share, most):
    rng = np.random.default_rng(17)
    rc = W.LJ_AR.rc if pot == "lj" else W.CU_LIKE.rc
    a = ratio * rc
    x = W.fcc_lattice(5, 5, 6, a)
    x = x[rng.permutation(len(x))[:int(share * len(x))]]
    x = x + rng.normal(0, 0.01, size=x.shape) + 0.25 * a
    L = a * np.array([5.0, 5.0, 6.0])
    v = rng.normal(0, 1e-3, size=x.shape)
    got = []
    for T in [t for t in (1, 2, 4, 8, 32) if 8 * t >= most]:
        if pot == "lj":
            ctx = lj_ctx(mdk, x, [0] * 3, L, [1] * 3, "mixed", v=v)
        else:
            ctx = eam_ctx(mdk, x, [0] * 3, L, [1] * 3, "mixed", W.tabulate_fs_eam(W.CU_LIKE), v=v)
        ctx.set_launch(T, 256)
        n = ctx.neighbor_counts()
        assert n.max() <= most and n.max() > most // 2
        r = list(ctx.compute())
        ctx.step(1.0, 12)
        got.append(r + list(ctx.get_state()) + list(ctx.compute()))
        ctx.close()
    for g in got[1:]:
        for p, q in zip(g, got[0]):
            assert np.array_equal(p, q)
