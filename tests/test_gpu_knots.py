"""Knot updates from device tensors (mdk_update_eam_knots) against the host
path: the same energies, forces and virials bit for bit, also after a new
workspace (which is filled from the host copy) and from another stream; other
sizes, or no workspace yet, are refused and change nothing."""
import numpy as np
import pytest

from paper_2511_22951_gb300 import workloads as W

from test_gpu_parity import eam_ctx

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


def system():
    rng = np.random.default_rng(2)
    x = W.fcc_lattice(4, 4, 5, 3.6) + rng.normal(0, 0.05, (320, 3))
    L = np.array([14.4, 14.4, 18.0])
    return np.mod(x, L), L


def scaled(t, f):
    return W.EAMTables(rc=t.rc, phi=f * t.phi, rho=t.rho / f, rho_max=t.rho_max, F=(2 - f) * t.F)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("side", [False, True])
def test_device_knots_equal_host_knots(mdk, prec, side):
    import torch
    x, L = system()
    t0 = W.tabulate_fs_eam(W.CU_LIKE, 2000, 1500)
    t1 = scaled(t0, 1.1)
    ref = eam_ctx(mdk, x, [0] * 3, L, [1] * 3, prec, t1)
    want = ref.compute()
    ctx = eam_ctx(mdk, x, [0] * 3, L, [1] * 3, prec, t0)
    ctx.compute()
    st = torch.cuda.Stream() if side else torch.cuda.current_stream()
    with torch.cuda.stream(st):
        k = [torch.tensor(q, device="cuda") for q in (t1.phi, t1.rho, t1.F)]
    ctx.stream.wait_stream(st)
    assert ctx.update_eam_knots(*k, t1.rc, t1.rho_max)
    for p, q in zip(ctx.compute(), want):
        assert np.array_equal(p, q)
    ctx.alloc_workspace()
    for p, q in zip(ctx.compute(), want):
        assert np.array_equal(p, q)
    short = [q[:-1].contiguous() for q in k]
    assert not ctx.update_eam_knots(*short, t1.rc, t1.rho_max)
    for p, q in zip(ctx.compute(), want):
        assert np.array_equal(p, q)
    ctx.close()
    ref.close()


def test_refused_without_workspace_or_eam(mdk):
    import torch
    x, L = system()
    k = [torch.ones(2000, dtype=torch.float64, device="cuda") for _ in range(3)]
    ctx = mdk.Context([0] * 3, L, [1] * 3, np.full(320, W.MASS_CU), "mixed")
    assert not ctx.update_eam_knots(*k, 5.5, 100.0)
    ctx.set_potential_lj(W.LJ_AR.eps, W.LJ_AR.sigma, 5.5, 1)
    ctx.set_state(x)
    assert not ctx.update_eam_knots(*k, 5.5, 100.0)
    ctx.close()
