"""What a knot update from the device refuses before anything is enqueued:
tensors that a kernel could not read as they are (host memory, another type, a
stride, another rank), tables of unequal length, and a stream under capture,
whose host copy would not hold the knots.  The potential stays as it was; the
differentiable function refuses capture as it did with knots from the host."""
import numpy as np
import pytest

from paper_2511_22951_gb300 import workloads as W

from test_gpu_parity import eam_ctx

pytestmark = pytest.mark.gpu


def system():
    rng = np.random.default_rng(2)
    x = W.fcc_lattice(4, 4, 5, 3.6) + rng.normal(0, 0.05, (320, 3))
    L = np.array([14.4, 14.4, 18.0])
    return np.mod(x, L), L


def test_tensors_a_kernel_cannot_read(mdk):
    import torch
    x, L = system()
    tab = W.tabulate_fs_eam(W.CU_LIKE, 2000, 1500)
    ctx = eam_ctx(mdk, x, [0] * 3, L, [1] * 3, "fp64", tab)
    want = ctx.compute()
    k = [torch.tensor(2.0 * q, device="cuda") for q in (tab.phi, tab.rho, tab.F)]
    wide = [torch.stack([q, q], 1)[:, 0] for q in k]        # same values, stride 2
    for n in range(3):
        for bad in (k[n].cpu(), k[n].float(), wide[n], k[n].reshape(1, -1)):
            with pytest.raises(ValueError):
                ctx.update_eam_knots(*[bad if m == n else k[m] for m in range(3)], tab.rc, tab.rho_max)
    with pytest.raises(ValueError):
        ctx.update_eam_knots(k[0], k[1][:-1].contiguous(), k[2], tab.rc, tab.rho_max)
    for p, q in zip(ctx.compute(), want):
        assert np.array_equal(p, q)
    ctx.close()


def test_stream_under_capture(mdk):
    import torch
    x, L = system()
    tab = W.tabulate_fs_eam(W.CU_LIKE, 2000, 1500)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        ctx = mdk.Context([0] * 3, L, [1] * 3, np.full(320, W.MASS_CU), "fp64", stream=st)
        ctx.set_potential_eam(tab)
        ctx.plan(tab.rc, 0.3)
        ctx.set_state(x, np.zeros_like(x))
        ctx.build_neighbors(tab.rc, 0.3)
        k = [torch.tensor(q, device="cuda") for q in (tab.phi, tab.rho, tab.F)]
        assert ctx.update_eam_knots(*k, tab.rc, tab.rho_max)
        want = ctx.compute()
        k2 = [2.0 * q for q in k]
        st.synchronize()
        g = torch.cuda.CUDAGraph()
        one = torch.zeros(1, device="cuda")
        with torch.cuda.graph(g, stream=st):
            one += 1.0
            assert not ctx.update_eam_knots(*k2, tab.rc, tab.rho_max)
        for p, q in zip(ctx.compute(), want):
            assert np.array_equal(p, q)
        ctx.alloc_workspace()                     # filled from the host copy
        for p, q in zip(ctx.compute(), want):
            assert np.array_equal(p, q)
    ctx.close()
