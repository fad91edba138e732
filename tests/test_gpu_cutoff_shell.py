"""Ideal lattices with a neighbour shell exactly at the cutoff, FP64.  Rounding
decides which pairs of that shell are inside; every kernel has to decide a
pair alike from both its atoms (the potentials jump at rc here), so that
forces come in opposite pairs: the net force is zero to the rounding of its
sum, N (number of neighbours) 2^-53 max|f_pair| at most, where one pair that
acts on one atom only leaves |V'(rc)|, ten orders more.  Half and full lists
decide alike: the energies agree to rounding."""
import ctypes

import numpy as np
import pytest

from paper_2511_22951_gb300 import workloads as W

from test_gpu_parity import eam_ctx, lj_ctx

pytestmark = pytest.mark.gpu


# lattice constant, shell (rc = a sqrt(shell / 2)), offset of the lattice
CASES = [(5.26, 4, 0.3), (5.13, 5, 1.7), (5.4, 4, 0.11)]
NEIGH = 100          # more than the neighbours of the fifth shell


def lattice(a, off):
    x = W.fcc_lattice(5, 5, 6, a) + off
    L = a * np.array([5.0, 5.0, 6.0])
    return np.mod(x, L), L


def check_net(F, fmax, jump):
    bound = len(F) * NEIGH * 2.0 ** -53 * fmax
    assert bound < 1e-3 * jump
    assert np.max(np.abs(F.sum(0))) <= bound


def shapes():
    return [("full", t) for t in (1, 2, 4, 8, 32)] + [("half", 1)]


@pytest.mark.parametrize("a,shell,off", CASES)
def test_lj(mdk, a, shell, off):
    x, L = lattice(a, off)
    rc = a * np.sqrt(shell / 2)
    eps, sig = W.LJ_AR.eps, W.LJ_AR.sigma
    f = lambda r: abs(24 * eps * (2 * (sig / r) ** 12 - (sig / r) ** 6) / r)  # noqa: E731
    fmax = max(f(a / np.sqrt(2)), f(a))
    E = []
    for kind, T in shapes():
        ctx = lj_ctx(mdk, x, [0] * 3, L, [1] * 3, "fp64", rc=rc, mode=0)
        ctx.set_list_kind(kind)
        ctx.set_launch(T, 128)
        e, F, _ = ctx.compute()
        ctx.close()
        check_net(F, fmax, f(rc))
        E.append(e[0])
    assert np.ptp(E) <= 1e-12 * abs(E[0])


@pytest.mark.parametrize("a,shell,off", CASES)
def test_eam(mdk, a, shell, off):
    x, L = lattice(a, off)
    rc = a * np.sqrt(shell / 2)
    r = np.linspace(0.0, rc, 1000)
    rho = 2.0 - r / rc
    F = -np.sqrt(np.linspace(0.0, 400.0, 1000) + 1.0)
    tab = W.EAMTables(rc=rc, phi=np.exp(-r), rho=rho, rho_max=400.0, F=F)
    fmax = np.exp(-a / np.sqrt(2)) + 1.0 / rc          # |F'| <= 1/2 at each end
    jump = np.exp(-rc)
    E = []
    for kind, T in shapes():
        ctx = eam_ctx(mdk, x, [0] * 3, L, [1] * 3, "fp64", tab)
        ctx.set_list_kind(kind)
        ctx.set_launch(T, 128)
        e, F, _ = ctx.compute()
        ctx.close()
        check_net(F, fmax, jump)
        E.append(e[0])
    assert np.ptp(E) <= 1e-12 * abs(E[0])


@pytest.mark.parametrize("a,shell,off", CASES)
def test_noalloc(mdk, a, shell, off):
    import torch
    x, L = lattice(a, off)
    rc = a * np.sqrt(shell / 2)
    eps, sig = W.LJ_AR.eps, W.LJ_AR.sigma
    f = lambda r: abs(24 * eps * (2 * (sig / r) ** 12 - (sig / r) ** 6) / r)  # noqa: E731
    P = ctypes.c_void_p
    xd = torch.tensor(x, device="cuda")
    F = torch.empty_like(xd)
    E = torch.empty(1, dtype=torch.float64, device="cuda")
    lo, per = np.zeros(3), np.ones(3, dtype=np.int32)
    r = mdk.load().mdk_lj_compute_noalloc(
        P(xd.data_ptr()), len(x), lo.ctypes.data_as(P), L.ctypes.data_as(P), per.ctypes.data_as(P),
        eps, sig, rc, 0, P(F.data_ptr()), P(E.data_ptr()),
        P(torch.cuda.current_stream().cuda_stream))
    assert r == 0
    check_net(F.cpu().numpy(), max(f(a / np.sqrt(2)), f(a)), f(rc))
