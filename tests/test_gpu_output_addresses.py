"""mdk_compute(on_device) takes E and the virial at every address that a device
copy reaches: in one system and in a batch, at 8-byte aligned device memory (the
sums' kernel stores there), at device memory off that alignment and in pinned
host memory; each gives the same bits."""
import ctypes

import numpy as np
import pytest

from paper_2511_22951_gb300 import workloads as W

pytestmark = pytest.mark.gpu

P = ctypes.c_void_p


def place(torch, where, n):
    """(address, reader) of n doubles."""
    if where == "pinned":
        t = torch.full((8 * n,), 7, dtype=torch.uint8).pin_memory()
        return t.data_ptr(), lambda: t.numpy().tobytes()
    off = int(where)
    t = torch.full((8 * n + 16,), 7, dtype=torch.uint8, device="cuda")
    return t.data_ptr() + off, lambda: t.cpu().numpy()[off:off + 8 * n].tobytes()


@pytest.mark.parametrize("sizes", [(5,), (4, 5, 6)])
@pytest.mark.parametrize("e_at,w_at", [("0", "0"), ("4", "0"), ("0", "4"), ("1", "3"), ("pinned", "0"),
                                       ("0", "pinned"), ("8", "pinned")])
def test_same_bits_at_every_address(mdk, sizes, e_at, w_at):
    import torch
    rng = np.random.default_rng(7)
    rs = [W.lattice_system(rng, (k, k, k), 5.26, W.MASS_AR, 0.0, sigma_jitter=0.05) for k in sizes]
    ctx = mdk.Context([r.lo for r in rs], [r.hi for r in rs], [r.periodic for r in rs],
                      np.concatenate([r.masses for r in rs]), "fp64", n_atoms=[r.n for r in rs])
    ctx.set_potential_lj(W.LJ_AR.eps, W.LJ_AR.sigma, W.LJ_AR.rc, 1)
    ctx.plan(W.LJ_AR.rc, 0.3)
    ctx.set_state(np.concatenate([r.x for r in rs]))
    E, _, Wv = ctx.compute()
    pe, re = place(torch, e_at, len(rs))
    pw, rw = place(torch, w_at, 6 * len(rs))
    assert mdk.load().mdk_compute(ctx.h, P(pe), None, P(pw), 1) == 0
    torch.cuda.synchronize()
    assert re() == E.tobytes() and rw() == Wv.tobytes()
    ctx.close()


def test_captured_by_the_caller(mdk):
    """A caller's graph holds the evaluation and writes E and W on replay."""
    import torch
    rng = np.random.default_rng(8)
    r = W.lattice_system(rng, (5, 5, 5), 5.26, W.MASS_AR, 0.0, sigma_jitter=0.05)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        ctx = mdk.Context(r.lo, r.hi, r.periodic, r.masses, "fp64", stream=st)
        ctx.set_potential_lj(W.LJ_AR.eps, W.LJ_AR.sigma, W.LJ_AR.rc, 1)
        ctx.plan(W.LJ_AR.rc, 0.3)
        ctx.set_state(r.x)
        E, F, Wv = ctx.compute()
        e = torch.zeros(1, dtype=torch.float64, device="cuda")
        w = torch.zeros(6, dtype=torch.float64, device="cuda")
        st.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            ctx.compute_device(e, None, w)
        assert float(e) == 0.0
        g.replay()
        st.synchronize()
    assert np.array_equal(e.cpu().numpy(), E) and np.array_equal(w.cpu().numpy(), Wv[0])
    ctx.close()
