"""mdk_lj_compute_noalloc at the ends of its sizes: the largest number of atoms
(every block of the force kernel has its own energy word), one block and one
atom more, and a single atom, against the FP64 evaluation of a context (1e-12,
the FP64 bar)."""
import ctypes

import numpy as np
import pytest

from paper_2511_22951_gb300 import workloads as W

from test_gpu_parity import lj_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cells,take", [((16, 32, 16), 32768), ((4, 4, 4), 16), ((4, 4, 4), 17), ((4, 4, 4), 1)])
def test_sizes(mdk, cells, take):
    import torch
    rng = np.random.default_rng(2)
    a, lj = 5.26, W.LJ_AR
    x = W.fcc_lattice(*cells, a)[:take] + rng.normal(0, 0.05, (take, 3))
    L = a * np.array(cells, dtype=float)
    x = np.mod(x, L)
    ctx = lj_ctx(mdk, x, [0] * 3, L, [1] * 3, "fp64")
    e, f, _ = ctx.compute()
    ctx.close()
    P = ctypes.c_void_p
    xd = torch.tensor(x, device="cuda")
    F = torch.full_like(xd, 7.0)
    E = torch.full((1,), 7.0, dtype=torch.float64, device="cuda")
    lo, per = np.zeros(3), np.ones(3, dtype=np.int32)
    assert mdk.load().mdk_lj_compute_noalloc(
        P(xd.data_ptr()), take, lo.ctypes.data_as(P), L.ctypes.data_as(P), per.ctypes.data_as(P), lj.eps,
        lj.sigma, lj.rc, 1, P(F.data_ptr()), P(E.data_ptr()),
        P(torch.cuda.current_stream().cuda_stream)) == 0
    assert abs(E.item() - e[0]) <= 1e-12 * abs(e[0]) + 1e-300
    assert np.max(np.abs(F.cpu().numpy() - f)) <= 1e-12 * np.max(np.abs(f)) + 1e-13
