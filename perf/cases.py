"""The work that a user of the MD library has it do, as timed cases.

Every case goes through the public entry points (the Context binding, the C
ABI functions under their own names, the differentiable EAM function).  The
sizes are those of this repository's workloads, tests and benchmark, plus
ragged lattices of the same materials:

  md        a trajectory segment as a restart script runs it: positions and
            velocities of a stored frame go in, the lists are built, `steps`
            velocity-Verlet steps run, the new frame and the energy and virial
            come back
  point     one energy / force / virial evaluation of new positions (list build
            included), as a relaxation or a sampling driver asks for it
  noalloc   the same for callers that may not allocate device memory
  isotherms the batched volume-temperature grid of the Hugoniot construction,
            each replica with its own thermostat
  train     a batch of compressed cells, the loss of its energies and forces and
            the gradient with respect to the potential's knots (table fitting)
  shock     a free slab driven by a rigid piston, and the profiles along x

The mixed path's pair arithmetic is FP32, so a program keeps its velocities,
forces, virials and knot parameters in single precision; positions and
energies stay in FP64.  The FP64 path's results are all FP64.
"""
import math

import numpy as np
import torch

from paper_2511_22951_gb300 import mdk
from paper_2511_22951_gb300 import workloads as W
from paper_2511_22951_gb300.adjoint import eam_energy_forces

KB = W.K_B
ACC = W.EV_PER_A_U_TO_A_PER_FS2
DEV = "cuda"


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------
def _md(name, pot, prec, cells, steps, outer=0.0, langevin=False):
    c = {"kind": "md", "pot": pot, "prec": prec, "nx": cells[0], "ny": cells[1],
         "nz": cells[2], "steps": steps, "outer": outer, "langevin": langevin}
    return dict(c, name=name) if name else c


def listed():
    return [
        # smallest run: a few hundred atoms, where launches and latency count
        _md("lj_fp64_256_run", "lj", "fp64", (4, 4, 4), 100),
        # a single evaluation inside another program's loop, no allocation
        {"name": "lj_noalloc_4000", "kind": "noalloc", "nx": 10, "ny": 10, "nz": 10},
        # an everyday system size
        _md("lj_mixed_32k_run", "lj", "mixed", (20, 20, 20), 100),
        # the benchmark's argon crystal, with its two-level lists
        _md("lj_mixed_8m_run", "lj", "mixed", (128, 128, 128), 50, outer=2.1),
        # NVT run of an uneven box
        _md("lj_mixed_nvt_ragged", "lj", "mixed", (61, 43, 37), 50, langevin=True),
        # the FP64 path on a large crystal
        _md("lj_fp64_500k_run", "lj", "fp64", (50, 50, 50), 10),
        # the aluminium bulk workload on the FP64 path
        _md("eam_fp64_256k_run", "eam", "fp64", (40, 40, 40), 10),
        # one evaluation of a small uneven metal cell
        {"name": "eam_mixed_point_ragged", "kind": "point", "pot": "eam", "prec": "mixed",
         "nx": 13, "ny": 17, "nz": 11},
        # the shock slab with its piston, then the profiles
        {"name": "eam_mixed_shock_slab", "kind": "shock", "prec": "mixed", "nx": 400, "nyz": 20,
         "steps": 40, "bins": 200},
        # table fitting on the 64 replicas of the cold curve
        {"name": "eam_mixed_cold_curve_train", "kind": "train", "prec": "mixed", "rep": 64,
         "nmin": 3, "nmax": 12},
        # the 8 x 8 isotherm grid
        {"name": "lj_mixed_isotherms", "kind": "isotherms", "prec": "mixed", "nv": 8, "nt": 8,
         "n": 12, "steps": 40},
        # the neural-network potential on the aluminium lattice
        _md("bpnn_mixed_131k_run", "bpnn", "mixed", (32, 32, 32), 2),
    ]


def _logint(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _box(rng, lo, hi):
    """Three cell counts, uneven, whose geometric mean is spread over [lo, hi]."""
    m = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    f = [rng.uniform(0.75, 1.3) for _ in range(3)]
    return tuple(max(int(lo), min(int(hi), int(round(m * q)))) for q in f)


def draw(rng):
    kind = rng.choice(["md", "md", "md", "md", "point", "noalloc", "shock", "train", "isotherms"])
    if kind == "md":
        pot, prec = rng.choice([("lj", "mixed"), ("lj", "mixed"), ("lj", "fp64"),
                                ("eam", "mixed"), ("eam", "fp64"), ("bpnn", "mixed")])
        if pot == "bpnn":
            return _md(None, pot, prec, _box(rng, 4, 30), rng.randint(2, 3))
        cells = _box(rng, 4, 110 if (pot, prec) == ("lj", "mixed") else 48)
        big = cells[0] * cells[1] * cells[2] > 60000
        steps = rng.randint(5, 10) if prec == "fp64" and big else rng.randint(20, 50 if big else 100)
        outer = 2.1 if pot == "lj" and prec == "mixed" and big and rng.random() < 0.5 else 0.0
        return _md(None, pot, prec, cells, steps, outer, rng.random() < 0.3)
    if kind == "point":
        pot, prec = rng.choice([("lj", "mixed"), ("lj", "fp64"), ("eam", "mixed"), ("eam", "fp64")])
        b = _box(rng, 4, 60)
        return {"kind": "point", "pot": pot, "prec": prec, "nx": b[0], "ny": b[1], "nz": b[2]}
    if kind == "noalloc":
        b = _box(rng, 4, 20)
        return {"kind": "noalloc", "nx": b[0], "ny": b[1], "nz": b[2]}
    if kind == "shock":
        return {"kind": "shock", "prec": rng.choice(["mixed", "mixed", "fp64"]),
                "nx": _logint(rng, 40, 400), "nyz": rng.randint(4, 20),
                "steps": rng.randint(10, 40), "bins": rng.randint(20, 250)}
    if kind == "train":
        lo = rng.randint(3, 5)
        return {"kind": "train", "prec": rng.choice(["mixed", "mixed", "fp64"]),
                "rep": _logint(rng, 4, 64), "nmin": lo, "nmax": rng.randint(lo + 1, 12)}
    return {"kind": "isotherms", "prec": "mixed", "nv": rng.randint(2, 8), "nt": rng.randint(2, 8),
            "n": rng.randint(6, 12), "steps": rng.randint(20, 40)}


# --------------------------------------------------------------------------
# inputs (on the GPU, from the seed)
# --------------------------------------------------------------------------
LATTICE = {"lj": (5.26, W.MASS_AR, 80.0, 2.0), "eam": (4.05, W.MASS_AL, 300.0, 1.0),
           "bpnn": (4.05, W.MASS_AL, 300.0, 1.0)}   # a, mass, T, dt
SKIN = 0.3
JITTER = {"lj": 0.10, "eam": 0.05, "bpnn": 0.05}    # thermal displacements (A)
U_P = 0.015                                          # piston speed (A/fs)
_TABLES = {}


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _tables(metal):
    if metal not in _TABLES:
        _TABLES[metal] = W.tabulate_fs_eam(W.AL_LIKE if metal == "al" else W.CU_LIKE)
    return _TABLES[metal]


def _lattice(g, nx, ny, nz, a, jitter):
    """Jittered FCC positions a quarter cell inside the box."""
    basis = torch.tensor([[0, 0, 0], [0.5, 0.5, 0], [0.5, 0, 0.5], [0, 0.5, 0.5]],
                         dtype=torch.float64, device=DEV)
    ax = [torch.arange(n, dtype=torch.float64, device=DEV) for n in (nz, ny, nx)]
    iz, iy, ix = torch.meshgrid(*ax, indexing="ij")
    cells = torch.stack([ix.reshape(-1), iy.reshape(-1), iz.reshape(-1)], 1)
    x = ((cells[:, None, :] + basis[None]).reshape(-1, 3) + 0.25) * a
    return x + jitter * torch.randn(x.shape, generator=g, dtype=torch.float64, device=DEV)


def _maxwell(g, n, mass, T):
    v = torch.randn((n, 3), generator=g, dtype=torch.float64, device=DEV)
    v *= math.sqrt(KB * T / mass * ACC)
    return v - v.mean(0)


def _system(case, seed):
    """x, v, box lengths and masses of a single-system case."""
    g = _gen(seed)
    pot = "lj" if case["kind"] == "noalloc" else "eam" if case["kind"] == "shock" else case["pot"]
    a, mass, T, dt = LATTICE[pot]
    n = (case["nx"], case["nyz"], case["nyz"]) if case["kind"] == "shock" else \
        (case["nx"], case["ny"], case["nz"])
    x = _lattice(g, *n, a, JITTER[pot])
    return {"x": x, "v": _maxwell(g, x.shape[0], mass, T), "a": a, "mass": mass, "T": T, "dt": dt,
            "L": [q * a for q in n], "pot": pot}


def _potential(ctx, pot):
    if pot == "lj":
        ctx.set_potential_lj(W.LJ_AR.eps, W.LJ_AR.sigma, W.LJ_AR.rc, W.LJ_AR.shift_mode)
        return W.LJ_AR.rc
    if pot == "eam":
        ctx.set_potential_eam(_tables("al"))
        return W.AL_LIKE.rc
    m = W.maise_like_bpnn(0, rc=6.0)
    ctx.set_potential_bpnn(m)
    return m.rc


def _outputs(ctx, n, reps=1):
    f = lambda *s: torch.empty(s, dtype=torch.float64, device=DEV)  # noqa: E731
    return {"ctx": ctx, "xo": f(n, 3), "vo": f(n, 3), "E": f(reps), "F": f(n, 3), "W": f(reps, 6)}


def _cold_curve(case, seed):
    """Uneven Cu-like FCC replicas: per-replica lattice constant and size."""
    rng = np.random.default_rng(int(seed))
    a = rng.uniform(3.0, 4.2, size=case["rep"])
    # sizes evenly over the range in a random order, so the batch's work does not depend on the seed
    span = case["nmax"] - case["nmin"] + 1
    n = case["nmin"] + rng.permutation(case["rep"]) % span
    g = _gen(seed)
    xs = []
    for q, m in zip(a, n):
        x = _lattice(g, int(m), int(m), int(m), float(q), 0.05)
        xs.append(torch.remainder(x, float(m) * float(q)))
    L = [[float(m) * float(q)] * 3 for q, m in zip(a, n)]
    return xs, L


def _knots():
    """Starting knots of the fit, single precision as a training program holds them."""
    t = _tables("cu")
    return [torch.tensor(k, dtype=torch.float32, device=DEV) for k in (t.phi, t.rho, t.F)]


def _isotherm_grid(case):
    """Lattice constants (v/v0 from 1 to 0.3) and temperatures (300 K to 1e5 K, geometric)."""
    a = 5.26 * np.cbrt(np.linspace(1.0, 0.3, case["nv"]))
    T = np.geomspace(300.0, 1e5, case["nt"])
    return a, T


def _isotherm_state(case, seed):
    a, T = _isotherm_grid(case)
    g = _gen(seed)
    n, xs, vs, L = case["n"], [], [], []
    for ai in a:
        for Tj in T:
            xs.append(_lattice(g, n, n, n, float(ai), 0.02 * float(ai)))
            vs.append(_maxwell(g, xs[-1].shape[0], W.MASS_AR, float(Tj)))
            L.append([n * float(ai)] * 3)
    return xs, vs, L, np.tile(T, len(a))


BETA = 5e-4      # thermostat stiffness of the isotherms (1/fs)
DT_ISO = 0.1     # the paper's step at 1e5 K (fs)
NVT = (80.0, 1e-3)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "noalloc":
        s = _system(case, seed)
        lo, hi = np.zeros(3), np.array(s["L"])
        return {"kind": kind, "x": s["x"], "lo": lo, "hi": hi, "per": np.ones(3, dtype=np.int32),
                "F": torch.empty_like(s["x"]),
                "E": torch.empty(1, dtype=torch.float64, device=DEV)}
    if kind == "train":
        xs, L = _cold_curve(case, seed)
        n = [x.shape[0] for x in xs]
        R = len(xs)
        ctx = mdk.Context(np.zeros((R, 3)), np.array(L), np.ones((R, 3)),
                          np.full(sum(n), W.MASS_CU), case["prec"], n_atoms=n)
        ctx.set_potential_eam(_tables("cu"))
        ctx.plan(W.CU_LIKE.rc, SKIN)
        ctx.set_state(torch.cat(xs))
        ctx.build_neighbors(W.CU_LIKE.rc, SKIN)
        ctx.autotune()
        knots = [k.requires_grad_(True) for k in _knots()]
        g = _gen(seed + 1)
        ref = 0.1 * torch.randn((sum(n), 3), generator=g, dtype=torch.float64, device=DEV)
        return {"kind": kind, "ctx": ctx, "knots": knots, "ref": ref, "mixed": case["prec"] == "mixed"}
    if kind == "isotherms":
        xs, vs, L, T = _isotherm_state(case, seed)
        R, n = len(xs), [x.shape[0] for x in xs]
        ctx = mdk.Context(np.zeros((R, 3)), np.array(L), np.ones((R, 3)),
                          np.full(sum(n), W.MASS_AR), case["prec"], n_atoms=n)
        rc = _potential(ctx, "lj")
        ctx.plan(rc, SKIN)
        x, v = torch.cat(xs), torch.cat(vs)
        ctx.set_state(x, v)
        ctx.build_neighbors(rc, SKIN)
        ctx.set_langevin_replicas(T, BETA, seed=7)
        ctx.autotune()
        return dict(_outputs(ctx, x.shape[0], R), kind=kind, x=x, v=v, dt=DT_ISO,
                    steps=case["steps"], mixed=case["prec"] == "mixed")
    s = _system(case, seed)
    n = s["x"].shape[0]
    lo, hi, per = np.zeros(3), np.array(s["L"]), np.ones(3)
    if kind == "shock":  # free along x, room ahead for the slab
        per[0] = 0
        lo[0], hi[0] = -2.0 * s["a"], hi[0] + 40.0 * s["a"]
    ctx = mdk.Context(lo, hi, per, np.full(n, s["mass"]), case["prec"])
    rc = _potential(ctx, s["pot"])
    ctx.plan(rc, SKIN)
    if case.get("outer"):
        ctx.set_outer_skin(case["outer"])
    ctx.set_state(s["x"], s["v"])
    if kind == "shock":
        ctx.set_piston(U_P, (s["x"][:, 0] < 2.0 * s["a"]).cpu().numpy())
    if case.get("langevin"):
        ctx.set_langevin([(-1e9, 1e9, NVT[0] if s["pot"] == "lj" else s["T"], (0.0, 0.0, 0.0), NVT[1])],
                         seed=7)
    ctx.build_neighbors(rc, SKIN)
    ctx.autotune()
    out = dict(_outputs(ctx, n), kind=kind, x=s["x"], v=s["v"], dt=s["dt"],
               steps=case.get("steps", 0), mixed=case["prec"] == "mixed")
    if kind == "shock":
        out["bins"] = (case["bins"], case["nx"] * s["a"] / case["bins"], s["L"][1] * s["L"][2])
    return out


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------
def _kept(s, t):
    """Velocities, forces, virials: single precision on the mixed path (its pair arithmetic)."""
    return t.float() if s["mixed"] else t


def run(s):
    kind = s["kind"]
    if kind == "noalloc":
        lj = W.LJ_AR
        r = mdk.load().mdk_lj_compute_noalloc(
            s["x"].data_ptr(), s["x"].shape[0], s["lo"].ctypes.data, s["hi"].ctypes.data,
            s["per"].ctypes.data, lj.eps, lj.sigma, lj.rc, lj.shift_mode, s["F"].data_ptr(),
            s["E"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        if r:
            raise mdk.MDKError(r, "mdk_lj_compute_noalloc")
        return {"E": s["E"], "F": s["F"]}
    ctx = s["ctx"]
    if kind == "train":
        E, F = eam_energy_forces(ctx, *s["knots"], W.CU_LIKE.rc, W.CU_LIKE.rho_max)
        loss = E.sum() + ((F - s["ref"]) ** 2).sum()
        g = torch.autograd.grad(loss, s["knots"])
        return {"E": E.detach(), "F": _kept(s, F.detach()), "g_phi": g[0], "g_rho": g[1], "g_F": g[2]}
    if kind == "point":
        ctx.set_state(s["x"])
        ctx.compute_device(s["E"], s["F"], s["W"])
        return {"E": s["E"], "F": _kept(s, s["F"]), "W": _kept(s, s["W"])}
    ctx.set_state(s["x"], s["v"])
    ctx.step(s["dt"], s["steps"])
    r = ctx.lib.mdk_get_state(ctx.h, s["xo"].data_ptr(), s["vo"].data_ptr(), 1)
    if r:
        raise mdk.MDKError(r, "mdk_get_state")
    ctx.compute_device(s["E"], None, s["W"])
    out = {"x": s["xo"], "v": _kept(s, s["vo"]), "E": s["E"], "W": _kept(s, s["W"])}
    if kind == "shock":
        nb, w, area = s["bins"]
        out["profiles"] = ctx.profiles(0, 0.0, w, nb, area)
    return out


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------
PAIR_FLOPS = {"lj": 23.0, "eam": 62.0}   # per unordered pair inside the cutoff
BPNN_PAIRS = 1431                         # unordered neighbour pairs per atom (54 neighbours)


def _pairs(density, rc):
    return 0.5 * density * 4.0 / 3.0 * math.pi * rc ** 3


def _bpnn_flops(n=54, nY=6, nZ=4, nS=43, G=51):
    pair = (21 + 7 * nY + 12 * nZ + 2 * nS) + (50 + 30 * nY + 8 * nZ + 16 * nS)
    return 0.5 * n * (n - 1) * pair + 4 * (G * 10 + 100 + 10)


def work(case):
    """The inputs read once and the outputs written once; every step
    evaluates every unordered pair inside the cutoff (neural network: every
    neighbour pair of every atom) once."""
    kind = case["kind"]
    if kind == "train":
        span = case["nmax"] - case["nmin"] + 1
        n = sum(4 * (case["nmin"] + q % span) ** 3 for q in range(case["rep"]))
        pairs = n * _pairs(4.0 / 3.6 ** 3, W.CU_LIKE.rc)
        return {"bytes": n * (24 + 24 + 24) + 6 * 5000 * 4, "flops": pairs * (62.0 + 90.0)}
    if kind == "isotherms":
        a, T = _isotherm_grid(case)
        n = 4 * case["n"] ** 3
        pairs = sum(len(T) * n * _pairs(4.0 / float(q) ** 3, W.LJ_AR.rc) for q in a)
        N = n * len(a) * len(T)
        return {"bytes": N * (48 + 48),
                "flops": (case["steps"] + 2) * pairs * 23.0}
    pot = "lj" if kind == "noalloc" else "eam" if kind == "shock" else case["pot"]
    a = LATTICE[pot][0]
    n = 4 * case["nx"] * (case["nyz"] ** 2 if kind == "shock" else case["ny"] * case["nz"])
    if pot == "bpnn":
        force = n * _bpnn_flops()
    else:
        force = n * _pairs(4.0 / a ** 3, W.LJ_AR.rc if pot == "lj" else W.AL_LIKE.rc) * PAIR_FLOPS[pot]
    if kind in ("point", "noalloc"):
        return {"bytes": n * 48 + 56, "flops": force}
    return {"bytes": n * 96 + 56, "flops": (case["steps"] + 2) * force}


# --------------------------------------------------------------------------
# the same results in 64 bits, with plain torch
# --------------------------------------------------------------------------
def _neighbours(x, L, per, r):
    """Padded table [N, K] of neighbours within r (index N: none) and their
    image shifts [N, K] (3-digit base-3 code of n + 1)."""
    N, dev = x.shape[0], x.device
    Lt = torch.tensor(L, dtype=torch.float64, device=dev)
    # atoms and their images within r of the box
    gx, gi, gc = [x], [torch.arange(N, device=dev)], [torch.full((N,), 13, device=dev)]
    lo = x.min(0).values
    hi = x.max(0).values
    for nz in (-1, 0, 1):
        for ny in (-1, 0, 1):
            for nx in (-1, 0, 1):
                n = (nx, ny, nz)
                if n == (0, 0, 0) or any(n[d] and not per[d] for d in range(3)):
                    continue
                y = x + torch.tensor(n, dtype=torch.float64, device=dev) * Lt
                m = ((y > lo - r) & (y < hi + r)).all(1).nonzero()[:, 0]
                gx.append(y[m])
                gi.append(m)
                gc.append(torch.full((m.numel(),), (nx + 1) + 3 * (ny + 1) + 9 * (nz + 1), device=dev))
    gx, gi, gc = torch.cat(gx), torch.cat(gi), torch.cat(gc)
    org = lo - r * 1.0001
    h = r * 1.0001
    nc = torch.floor((hi + r * 1.0001 - org) / h).long() + 1
    c = torch.floor((gx - org) / h).long()
    cell = c[:, 0] + nc[0] * (c[:, 1] + nc[1] * c[:, 2])
    order = torch.argsort(cell)
    cs = cell[order]
    ncell = int(nc.prod())
    start = torch.searchsorted(cs, torch.arange(ncell + 1, device=dev))
    width = int((start[1:] - start[:-1]).max())
    gx, gi, gc = gx[order], gi[order], gc[order]
    off = [dx + int(nc[0]) * (dy + int(nc[1]) * dz)
           for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)]
    slot = torch.arange(width, device=dev)
    nb, code, K = [], [], 0
    chunk = max(1, int(6e7 / (27 * width)))
    own = cell[:N]
    for a in range(0, N, chunk):
        b = min(N, a + chunk)
        cc = own[a:b, None] + torch.tensor(off, device=dev)
        s0, s1 = start[cc], start[cc + 1]
        q = s0[:, :, None] + slot
        ok = q < s1[:, :, None]
        q = torch.where(ok, q, torch.zeros_like(q)).reshape(b - a, -1)
        d = gx[q] - x[a:b, None, :]
        r2 = (d * d).sum(2)
        me = torch.arange(a, b, device=dev)[:, None]
        ok = ok.reshape(b - a, -1) & (r2 < r * r) & ~((gi[q] == me) & (gc[q] == 13))
        k = int(ok.sum(1).max()) if b > a else 0
        # kept candidates first
        pos = torch.argsort((~ok).to(torch.int8), dim=1, stable=True)[:, :k]
        okk = torch.gather(ok, 1, pos)
        qq = torch.gather(q, 1, pos)
        nb.append(torch.where(okk, gi[qq], torch.full_like(qq, N)).to(torch.int32))
        code.append(torch.where(okk, gc[qq], torch.full_like(qq, 13)).to(torch.int8))
        K = max(K, k)
    pad = lambda t, v: torch.nn.functional.pad(t, (0, K - t.shape[1]), value=v)  # noqa: E731
    return torch.cat([pad(t, N) for t in nb]), torch.cat([pad(t, 13) for t in code])


class _Ref64:
    """Energies, forces and virials of one system in FP64."""

    MARGIN = 1.0  # the neighbour table holds pairs within rc + margin

    def __init__(self, pot, x, L, per=(1, 1, 1), knots=None):
        self.pot, self.L, self.per = pot, torch.tensor(L, dtype=torch.float64, device=x.device), per
        self.box, self.x0 = L, None
        if pot == "lj":
            self.rc = W.LJ_AR.rc
        elif pot == "bpnn":
            self.m = W.maise_like_bpnn(0, rc=6.0)
            self.rc = self.m.rc
        else:
            t = _tables("cu" if knots is not None else "al")
            self.rc, self.rho_max = t.rc, t.rho_max
            k = knots if knots is not None else \
                [torch.tensor(q, dtype=torch.float64, device=x.device) for q in (t.phi, t.rho, t.F)]
            self.tab = [(q, self._slopes(q)) for q in k]

    def _renew(self, x):
        """The table again once an atom has moved half the margin."""
        if self.x0 is None or float((x - self.x0).square().sum(1).max()) > (0.5 * self.MARGIN) ** 2:
            self.x0 = x.clone()
            self.nb, self.code = _neighbours(x, self.box, self.per, self.rc + self.MARGIN)

    @staticmethod
    def _slopes(y):
        """h times the knot slopes: 3-point differences."""
        return torch.cat([(0.5 * (-3 * y[0] + 4 * y[1] - y[2]))[None], 0.5 * (y[2:] - y[:-2]),
                          (0.5 * (3 * y[-1] - 4 * y[-2] + y[-3]))[None]])

    @staticmethod
    def _spline(tab, u, der):
        """Cubic Hermite value, or derivative with respect to u, at u knots."""
        y, m = tab
        k = u.detach().floor().long().clamp(0, y.shape[0] - 2)
        t = u - k
        y0, y1, m0, m1 = y[k], y[k + 1], m[k], m[k + 1]
        if der:
            return (6 * t * t - 6 * t) * (y0 - y1) + (3 * t * t - 4 * t + 1) * m0 + (3 * t * t - 2 * t) * m1
        t2, t3 = t * t, t * t * t
        return y0 + (3 * t2 - 2 * t3) * (y1 - y0) + (t3 - 2 * t2 + t) * m0 + (t3 - t2) * m1

    def _vec(self, x, a, b):
        xp = torch.cat([x, torch.full((1, 3), 1e18, dtype=torch.float64, device=x.device)])
        j = self.nb[a:b].long()
        code = self.code[a:b].long()
        q = torch.arange(27, device=x.device)
        n = torch.stack([q % 3 - 1, (q // 3) % 3 - 1, q // 9 - 1], 1) * self.L
        d = (xp[j] - x[a:b, None, :]) + n[code]
        return j, d, (d * d).sum(2)

    def _chunks(self, per_atom_bytes):
        N = self.x0.shape[0]
        c = max(1, int(12e9 / (self.nb.shape[1] * per_atom_bytes)))
        return [(a, min(N, a + c)) for a in range(0, N, c)]

    def forces(self, x):
        """(E, F [N, 3], W [6], U_i [N], W_i [N, 6])."""
        self._renew(x)
        if self.pot == "bpnn":
            return self._bpnn(x)
        if self.pot == "eam":
            dr = self.rc / (self.tab[0][0].shape[0] - 1)
            drho = self.rho_max / (self.tab[2][0].shape[0] - 1)
            rho = []
            for a, b in self._chunks(200):
                _, _, r2 = self._vec(x, a, b)
                ok = r2 < self.rc ** 2
                u = torch.sqrt(torch.where(ok, r2, torch.ones_like(r2))) / dr
                rho.append(torch.where(ok, self._spline(self.tab[1], u, False), torch.zeros_like(u)).sum(1))
            rho = torch.cat(rho)
            Fe = self._spline(self.tab[2], rho / drho, False)
            dF = self._spline(self.tab[2], rho / drho, True) / drho
            dFp = torch.cat([dF, dF.new_zeros(1)])
        F, U, Wi = [], [], []
        for a, b in self._chunks(400):
            j, d, r2 = self._vec(x, a, b)
            ok = r2 < self.rc ** 2
            r2 = torch.where(ok, r2, torch.full_like(r2, 4.0))
            d = torch.where(ok[:, :, None], d, torch.zeros_like(d))
            if self.pot == "lj":
                p = W.LJ_AR
                s6 = (p.sigma ** 2 / r2) ** 3
                c6 = (p.sigma / p.rc) ** 6
                e = 4 * p.eps * (s6 * s6 - s6) - 4 * p.eps * (c6 * c6 - c6)
                fr = -24 * p.eps * (2 * s6 * s6 - s6) / r2
            else:
                r = torch.sqrt(r2)
                e = self._spline(self.tab[0], r / dr, False)
                fr = (self._spline(self.tab[0], r / dr, True) +
                      (dF[a:b, None] + dFp[j]) * self._spline(self.tab[1], r / dr, True)) / dr / r
            fr = torch.where(ok, fr, torch.zeros_like(fr))
            f = fr[:, :, None] * d
            F.append(f.sum(1))
            U.append(0.5 * torch.where(ok, e, torch.zeros_like(e)).sum(1) +
                     (Fe[a:b] if self.pot == "eam" else 0.0))
            w = -0.5 * torch.stack([f[:, :, p] * d[:, :, q] for p, q in
                                    ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))], 2)
            Wi.append(w.sum(1))
        F, U, Wi = torch.cat(F), torch.cat(U), torch.cat(Wi)
        return U.sum(), F, Wi.sum(0), U, Wi

    def _bpnn(self, x):
        m, N = self.m, x.shape[0]
        t = lambda v: torch.tensor(v, dtype=torch.float64, device=x.device)  # noqa: E731
        W01, b1, W12, b2, w23 = t(m.W01), t(m.b1), t(m.W12), t(m.b2), t(m.w23)
        F = torch.zeros((N + 1, 3), dtype=torch.float64, device=x.device)
        U, Wi = [], []
        K = int((self.nb < N).sum(1).max())
        chunk = max(1, int(6e9 / (K * K * 8 * 60)))
        for a in range(0, N, chunk):
            b = min(N, a + chunk)
            j, d, r2 = self._vec(x, a, b)
            ok = r2 < m.rc ** 2
            pos = torch.argsort((~ok).to(torch.int8), dim=1, stable=True)[:, :int(ok.sum(1).max())]
            ok, j = torch.gather(ok, 1, pos), torch.gather(j, 1, pos)
            d = torch.gather(d, 1, pos[:, :, None].expand(-1, -1, 3))
            # absent neighbours: distinct far points, cut off
            far = 10.0 * m.rc * (1 + torch.arange(d.shape[1], device=x.device, dtype=torch.float64))
            d = torch.where(ok[:, :, None], d, far[None, :, None].expand_as(d)).detach().requires_grad_(True)
            r = torch.sqrt((d * d).sum(2))
            fc = torch.where(r < m.rc, 0.5 * (torch.cos(math.pi * r.clamp(max=m.rc) / m.rc) + 1), 0 * r)
            G = [(torch.exp(-p[0] * (r - p[1]) ** 2) * fc).sum(1) for p in m.rad_par]
            s = d[:, :, None, :] - d[:, None, :, :]
            rjk2 = (s * s).sum(3)
            eye = torch.eye(d.shape[1], dtype=torch.bool, device=x.device)
            rjk = torch.sqrt(torch.where(eye, torch.ones_like(rjk2), rjk2))
            up = torch.triu(torch.ones_like(eye), 1)
            near = up & (rjk < m.rc)
            fjk = torch.where(near, 0.5 * (torch.cos(math.pi * rjk.clamp(max=m.rc) / m.rc) + 1), 0 * rjk)
            f3 = fc[:, :, None] * fc[:, None, :] * fjk
            c = (d[:, :, None, :] * d[:, None, :, :]).sum(3) / (r[:, :, None] * r[:, None, :])
            q2 = (r * r)[:, :, None] + (r * r)[:, None, :] + rjk2
            pw = {}
            for eta in sorted(set(m.ang_par[:, 2])):
                Y = f3 * torch.exp(-eta * torch.where(f3 > 0, q2, torch.zeros_like(q2)))
                for k, (z, lam, et) in enumerate(m.ang_par):
                    if et == eta:
                        if (z, lam) not in pw:
                            pw[(z, lam)] = 2.0 ** (1 - z) * (1 + lam * c) ** int(z)
                        G.append((k, (pw[(z, lam)] * Y).sum((1, 2))))
            G = G[:m.n_rad] + [g for _, g in sorted(G[m.n_rad:], key=lambda q: q[0])]
            h = torch.tanh(torch.tanh(torch.stack(G, 1) @ W01 + b1) @ W12 + b2)
            e = h @ w23 + m.b3
            (g,) = torch.autograd.grad(e.sum(), d)
            g = torch.where(ok[:, :, None], g, torch.zeros_like(g))
            dd = d.detach()
            F.index_add_(0, j.reshape(-1), -g.reshape(-1, 3))
            F[a:b] += g.sum(1)
            dd = torch.where(ok[:, :, None], dd, torch.zeros_like(dd))
            U.append(e.detach())
            Wi.append(-torch.stack([(dd[:, :, p] * g[:, :, q]).sum(1) for p, q in
                                    ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))], 1))
            del G, pw, c, f3, q2, s, rjk, rjk2, e, g, d
        U, Wi = torch.cat(U), torch.cat(Wi)
        return U.sum(), F[:N], Wi.sum(0), U, Wi


def _mulhilo(a, b):
    """High and low words of the unsigned product of 64-bit words held in int64."""
    M = 0xFFFFFFFF
    a0, a1, b0, b1 = a & M, (a >> 32) & M, b & M, (b >> 32) & M
    p00, p01, p10 = a0 * b0, a0 * b1, a1 * b0
    mid = ((p00 >> 32) & M) + (p01 & M) + (p10 & M)
    return a1 * b1 + ((p01 >> 32) & M) + ((p10 >> 32) & M) + ((mid >> 32) & M), a * b


def _signed(v):
    return v - (1 << 64) if v >= (1 << 63) else v


def _noise(ids, step, seed):
    """xi - 1/2 [N, 3]: Philox4x64-10 (Salmon et al., SC 2011), counter (id, step), key (seed, 0)."""
    z = torch.zeros_like(ids)
    c = [ids.clone(), z + step, z.clone(), z.clone()]
    k0, k1 = seed, 0
    for r in range(10):
        if r:
            k0 = (k0 + 0x9E3779B97F4A7C15) & (2 ** 64 - 1)
            k1 = (k1 + 0xBB67AE8584CAA73B) & (2 ** 64 - 1)
        h0, l0 = _mulhilo(c[0], z + _signed(0xD2E7470EE14C6C93))
        h1, l1 = _mulhilo(c[2], z + _signed(0xCA5A826395121157))
        c = [h1 ^ c[1] ^ _signed(k0), l1, h0 ^ c[3] ^ _signed(k1), l0]
    out = torch.stack(c[:3], 1)
    return ((out >> 11) & ((1 << 53) - 1)).double() * 2.0 ** -53 - 0.5


def _trajectory(ref, x, v, mass, dt, steps, piston=None, thermostat=None, ids=None):
    """Velocity Verlet; thermostat = (T, beta): the Langevin force of every evaluation after the first."""
    c = 0.5 * dt * ACC / mass
    x, v = x.clone(), v.clone()

    def kick(f):
        v.add_(f, alpha=c)
        if piston is not None:
            v[piston] = torch.tensor([U_P, 0.0, 0.0], dtype=torch.float64, device=v.device)

    F = ref.forces(x)[1]
    for s in range(1, steps + 1):
        kick(F)
        x.add_(v, alpha=dt)
        F = ref.forces(x)[1]
        if thermostat is not None:
            T, beta = thermostat
            sig = math.sqrt(24 * beta * mass * KB * T / (dt * ACC))
            F = F + (-beta * mass / ACC) * v + sig * _noise(ids, s, 7)
        kick(F)
    return x, v


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        xs, L = _cold_curve(case, seed)
        knots = [k.double().requires_grad_(True) for k in _knots()]
        n = sum(x.shape[0] for x in xs)
        ref = 0.1 * torch.randn((n, 3), generator=_gen(seed + 1), dtype=torch.float64, device=DEV)
        Es, Fs, grads, o = [], [], None, 0
        for x, l in zip(xs, L):  # the loss is a sum over replicas
            E, F, _, _, _ = _Ref64("eam", x, l, knots=knots).forces(x)
            loss = E + ((F - ref[o:o + x.shape[0]]) ** 2).sum()
            g = torch.autograd.grad(loss, knots)
            grads = list(g) if grads is None else [p + q for p, q in zip(grads, g)]
            Es.append(E.detach())
            Fs.append(F.detach())
            o += x.shape[0]
        return {"E": torch.stack(Es), "F": torch.cat(Fs), "g_phi": grads[0], "g_rho": grads[1],
                "g_F": grads[2]}
    with torch.no_grad():
        if kind == "isotherms":
            xs, vs, L, T = _isotherm_state(case, seed)
            xo, vo, E, Wt, o = [], [], [], [], 0
            for x, v, l, Tj in zip(xs, vs, L, T):
                r = _Ref64("lj", x, l)
                ids = torch.arange(o, o + x.shape[0], device=DEV)
                x, v = _trajectory(r, x, v, W.MASS_AR, DT_ISO, case["steps"],
                                   thermostat=(float(Tj), BETA), ids=ids)
                e, _, w, _, _ = r.forces(x)
                xo.append(x)
                vo.append(v)
                E.append(e)
                Wt.append(w)
                o += x.shape[0]
            # positions may be wrapped at a list build: no value for them
            return {"x": None, "v": torch.cat(vo), "E": torch.stack(E), "W": torch.stack(Wt)}
        s = _system(case, seed)
        if s["pot"] != "bpnn" or kind != "md":
            r = _Ref64(s["pot"], s["x"], s["L"], (0, 1, 1) if kind == "shock" else (1, 1, 1))
        if kind in ("point", "noalloc"):
            E, F, w, _, _ = r.forces(s["x"])
            return {"E": E[None], "F": F} if kind == "noalloc" else {"E": E[None], "F": F, "W": w[None]}
    if s["pot"] == "bpnn":
        if s["x"].shape[0] * (case["steps"] + 2) > 6e5:
            return None  # over 20 seconds
        r = _Ref64("bpnn", s["x"], s["L"])
        x, v = _trajectory(r, s["x"], s["v"], s["mass"], s["dt"], case["steps"],
                           thermostat=(s["T"], NVT[1]) if case["langevin"] else None,
                           ids=torch.arange(s["x"].shape[0], device=DEV))
        E, _, w, _, _ = r.forces(x)
        return {"x": x, "v": v, "E": E[None], "W": w[None]}
    with torch.no_grad():
        if s["x"].shape[0] * (case["steps"] + 2) > 4.5e8:
            return None  # over 20 seconds
        piston = s["x"][:, 0] < 2.0 * s["a"] if kind == "shock" else None
        T = NVT[0] if s["pot"] == "lj" else s["T"]
        x, v = _trajectory(r, s["x"], s["v"], s["mass"], s["dt"], case["steps"], piston,
                           (T, NVT[1]) if case.get("langevin") else None,
                           torch.arange(s["x"].shape[0], device=DEV))
        E, _, w, U, Wi = r.forces(x)
        out = {"x": x, "v": v, "E": E[None], "W": w[None]}
        if kind == "shock":
            out["profiles"] = _profiles64(x, v, U, Wi, s["mass"], case["bins"],
                                          case["nx"] * s["a"] / case["bins"], s["L"][1] * s["L"][2])
        return out


def _profiles64(x, v, U, Wi, mass, nb, w, area):
    """N, M, u[3], T[3], E_pot, P[6], E_kin, V of every bin along x."""
    l = torch.floor(x[:, 0] / w).long()
    m = (l >= 0) & (l < nb)
    l, v, U, Wi = l[m], v[m], U[m], Wi[m]
    tot = lambda q: torch.zeros((nb,) + q.shape[1:], dtype=torch.float64, device=q.device).index_add_(0, l, q)  # noqa: E731
    N = tot(torch.ones_like(U))
    n1 = N.clamp(min=1)
    u = tot(v) / n1[:, None]
    du = v - u[l]
    k = mass / ACC * tot(torch.stack([du[:, p] * du[:, q] for p, q in
                                      ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))], 1))
    V = w * area
    return torch.cat([N[:, None], mass * N[:, None], u, k[:, :3] / (KB * n1[:, None]), tot(U)[:, None],
                      (k + tot(Wi)) / V, 0.5 * k[:, :3].sum(1, keepdim=True),
                      torch.full((nb, 1), V, dtype=torch.float64, device=v.device)], 1)
