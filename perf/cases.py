"""Timed workloads of the ETDM library: what its users have it evaluate.

Every case goes through the package's Python entry points.  The systems are the
recipes of ``etdm_synth`` (small molecules, boxes of water-like units, a batch of
uneven molecules, crystals with k-points) at the sizes of the tests and of the
benchmark; ``draw`` spreads the same recipes over the range between them.

``exact`` restates the model in plain torch FP64 (dense basis on the grid, the
analytic overlap and kinetic matrices, spectral Poisson solve, Slater exchange,
``torch.matrix_exp`` and automatic differentiation) and calls nothing of the
library.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

import etdm_synth as synth
from paper_2101_12597_gb300 import etdm

DEV = torch.device("cuda", 0)
F64 = torch.float64


# ---- cases --------------------------------------------------------------------

def listed():
    return [
        # the smallest call: one 8-atom molecule through the autograd Function
        # (energy in the forward pass, the adjoint in the backward pass), in the
        # default precision; launches and latency count
        dict(name="mol8_autograd_fp64", kind="point", recipe="atoms", units=8, box=6.4,
             gx=32, gy=32, gz=32, rcut=0.0, spread=0.05, geom=0, precision="fp64",
             entry="autograd"),
        # a whole calculation: ten minimization steps of the same molecule, one
        # synchronization per line-search trial
        dict(name="mol8_minimize_fp64", kind="minimize", recipe="atoms", units=8, box=6.4,
             gx=32, gy=32, gz=32, rcut=0.0, spread=0.05, geom=0, precision="fp64", steps=10),
        # two water-like units on a grid that is no multiple of a tile, from and
        # to host buffers (a caller without device arrays)
        dict(name="water2_ragged_host_mixed", kind="point", recipe="water", lx=2, ly=1, lz=1,
             box=6.0, gx=36, gy=28, gz=44, rcut=3.0, spread=0.05, geom=11, precision="mixed",
             entry="host"),
        # the liquid box of the paper's size (32 units) in the default precision ...
        dict(name="water32_fp64", kind="point", recipe="water", lx=4, ly=4, lz=2, box=9.9,
             gx=96, gy=96, gz=96, rcut=4.0, spread=0.02, geom=1, precision="fp64",
             entry="device"),
        # ... and in mixed precision
        dict(name="water32_mixed", kind="point", recipe="water", lx=4, ly=4, lz=2, box=9.9,
             gx=96, gy=96, gz=96, rcut=4.0, spread=0.02, geom=1, precision="mixed",
             entry="device"),
        # the largest box one GPU evaluates (the benchmark's default workload)
        dict(name="water576_mixed", kind="point", recipe="water", lx=9, ly=8, lz=8, box=25.0,
             gx=192, gy=192, gz=192, rcut=3.5, spread=0.01, geom=2, precision="mixed",
             entry="device"),
        # a set of uneven molecules evaluated together
        dict(name="molecules148_mixed", kind="batch", count=148, most=20, grid=48, spread=0.05,
             geom=3),
        # a small crystal over 2x2x2 k-points on a ragged grid: every launch short
        dict(name="crystal8_eig", kind="crystal", cx=2, cy=2, cz=2, spacing=2.6, exps=3, Z=1.5,
             gx=26, gy=24, gz=22, rcut=3.0, kmesh=2, spread=0.05, geom=8, expm="eig"),
        # a k-point calculation of the benchmark's size (M = 512, 8 k-points): the
        # exact gradient through the eigendecomposition.  Four Gaussians per atom,
        # as in the water boxes: the eight of the benchmark's crystal leave
        # eigenvalues of 1e-7 in S(k) and results that are defined to 1e-9 only
        dict(name="crystal128_eig", kind="crystal", cx=4, cy=4, cz=8, spacing=2.8, exps=4, Z=4.0,
             gx=56, gy=56, gz=112, rcut=4.0, kmesh=2, spread=0.01, geom=4, expm="eig"),
        # ... and scaling and squaring with the approximate gradient, at an odd size
        # (M = 500)
        dict(name="crystal125_ss", kind="crystal", cx=5, cy=5, cz=5, spacing=2.8, exps=4, Z=4.0,
             gx=70, gy=70, gz=70, rcut=4.0, kmesh=2, spread=0.01, geom=4, expm="ss"),
        # self-interaction correction of a molecule: one density, Poisson solve
        # and potential matrix per occupied orbital
        dict(name="mol8_pzsic", kind="sic", units=8, box=6.4, gx=32, gy=32, gz=32, spread=0.05,
             geom=0),
        # the stand-alone L-BFGS direction over the variables of the largest box
        dict(name="direction_5m", kind="direction", n=2304 * 2304, pairs=3),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _axis(n):
    """The nearest grid size whose prime factors are at most 13 (odd ones too)."""
    n = max(16, min(192, int(round(n))))
    while True:
        m = n
        for p in (2, 3, 5, 7, 11, 13):
            while m % p == 0:
                m //= p
        if m == 1:
            return n
        n += 1


def draw(rng):
    kind = rng.choice(["atoms", "water", "water", "batch", "crystal", "crystal", "sic",
                       "direction", "minimize"])
    geom = rng.randrange(1000)
    if kind in ("atoms", "minimize", "sic"):
        units = rng.choice([4, 6, 8, 10, 12])
        box = round(rng.uniform(5.6, 7.2), 2)
        g = [_axis(box / rng.uniform(0.16, 0.24)) for _ in range(3)]
        c = dict(units=units, box=box, gx=g[0], gy=g[1], gz=g[2], spread=0.05, geom=geom)
        if kind == "sic":
            return dict(kind="sic", **c)
        c.update(recipe="atoms", rcut=0.0, precision="fp64")
        if kind == "minimize":
            return dict(kind="minimize", steps=rng.randint(4, 12), **c)
        return dict(kind="point", entry=rng.choice(["device", "host", "autograd"]), **c)
    if kind == "water":
        units = _log(rng, 2, 120)
        edge = units ** (1.0 / 3.0)
        lx, ly, lz = (max(1, int(round(edge * f))) for f in
                      (rng.uniform(0.8, 1.3), rng.uniform(0.8, 1.3), rng.uniform(0.8, 1.3)))
        box = round(max(6.0, 3.13 * (lx * ly * lz) ** (1.0 / 3.0)), 2)
        h = rng.uniform(0.12, 0.2)
        return dict(kind="point", recipe="water", lx=lx, ly=ly, lz=lz, box=box,
                    gx=_axis(box / h), gy=_axis(box / h * rng.uniform(0.9, 1.1)),
                    gz=_axis(box / h * rng.uniform(0.9, 1.1)), rcut=rng.choice([3.0, 3.5]),
                    spread=0.02, geom=geom, precision=rng.choice(["mixed", "fp64"]),
                    entry=rng.choice(["device", "host", "autograd"]))
    if kind == "batch":
        return dict(kind="batch", count=int(_log(rng, 3, 148)), most=rng.randint(6, 20),
                    grid=rng.choice([45, 48]), spread=0.05, geom=geom)
    if kind == "crystal":
        cx, cy, cz = (rng.randint(2, 5) for _ in range(3))
        exps = rng.randint(2, 4)
        spacing = round(rng.uniform(2.6, 2.8), 2)
        h = rng.uniform(0.2, 0.22)
        return dict(kind="crystal", cx=cx, cy=cy, cz=cz, spacing=spacing, exps=exps, Z=2.0,
                    gx=_axis(cx * spacing / h), gy=_axis(cy * spacing / h),
                    gz=_axis(cz * spacing / h), rcut=3.0 if min(cx, cy, cz) < 3 else 4.0,
                    kmesh=rng.choice([1, 2]), spread=0.01, geom=geom,
                    expm=rng.choice(["eig", "ss"]))
    return dict(kind="direction", n=int(_log(rng, 16, 5_000_000)), pairs=rng.randint(1, 8))


# ---- inputs -------------------------------------------------------------------

def _systems(case):
    """The system dicts (geometry, basis, grid) of a case: its own, whatever the seed."""
    kind = case["kind"]
    if kind == "batch":
        return synth.molecule_batch(n_mol=case["count"], atoms=(2, case["most"]),
                                    grid=(case["grid"],) * 3, seed=case["geom"])
    grid = (case["gx"], case["gy"], case["gz"])
    if kind == "crystal":
        return [synth.crystal(cells=(case["cx"], case["cy"], case["cz"]),
                              spacing_ang=case["spacing"], n_exp=case["exps"], Z=case["Z"],
                              grid=grid, rcut_ang=case["rcut"], kmesh=case["kmesh"],
                              kT_ev=0.5, seed=case["geom"])]
    if kind == "sic" or case["recipe"] == "atoms":
        return [synth.random_atoms(n_atoms=case["units"], box_ang=case["box"], grid=grid,
                                   seed=case["geom"])]
    return [synth.water_box(lattice=(case["lx"], case["ly"], case["lz"]), box_ang=case["box"],
                            grid=grid, rcut_ang=case["rcut"], seed=case["geom"])]


def _sizes(d):
    M, N = len(d["bf_exp"]), d["n_electrons"] // 2
    return M, N, M - N


def _variables(case, systems, seed):
    """Seeded variables: packed A_ov of every system, or the M^2 reals of every A(k)."""
    n = 0
    for d in systems:
        M, N, V = _sizes(d)
        n += M * M * len(d["kw"]) if case["kind"] == "crystal" else \
            M * M if case["kind"] == "sic" else N * V
    return np.random.default_rng(seed).normal(0.0, case["spread"], size=n)


def _bloch(d, kind):
    """k-points and weights of the full-A cases (the Gamma point for PZ-SIC)."""
    if kind == "sic":
        return np.zeros((1, 3)), np.ones(1)
    return d["kpts"], d["kw"]


def _full_reference(d, kind):
    """C0(k) = S(k)^(-1/2) and occupations (n_k, M): what a calculation restarted
    from stored orbitals hands over.  Integer occupation for PZ-SIC, else a
    Fermi edge a few orbitals wide, cut to zero in its tail."""
    kpts, kw = _bloch(d, kind)
    M, N, _ = _sizes(d)
    C0 = []
    for k in kpts:
        S, _ = _overlap_kinetic(d, k)
        w, Q = torch.linalg.eigh(S)
        C0.append((Q / w.sqrt()) @ Q.conj().T)
    level = np.arange(M, dtype=np.float64)
    f = np.where(level < N, 1.0, 0.0)
    if kind == "crystal":
        f = 1.0 / (1.0 + np.exp(np.clip((level - N + 0.5) / 2.0, -40.0, 40.0)))
        f[f < 1e-6] = 0.0
        f *= N / f.sum()
    return C0, np.stack([2.0 * w * f for w in kw])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "direction":
        n, m = case["n"], case["pairs"]
        r = torch.Generator(device=DEV)
        r.manual_seed(int(seed))
        S = 0.1 * torch.randn((m, n), dtype=F64, device=DEV, generator=r)
        # curvature between 0.5 and 2 along every variable: y.s > 0
        Y = S * (0.5 + 1.5 * torch.rand((1, n), dtype=F64, device=DEV, generator=r))
        g = torch.randn(n, dtype=F64, device=DEV, generator=r)
        h0 = 0.3 + torch.rand(n, dtype=F64, device=DEV, generator=r)
        return dict(case=case, g=g, S=S, Y=Y, h0=h0, p=torch.empty_like(g))
    systems = _systems(case)
    host = _variables(case, systems, seed)
    if kind == "batch":
        solver = etdm.ETDMBatch(systems, precision="mixed")
        return dict(case=case, solver=solver, a=torch.tensor(host, device=DEV))
    d = systems[0]
    if kind == "crystal":
        solver = etdm.ETDM(d, expm=case["expm"])
    elif kind == "sic":
        solver = etdm.ETDM(d, param="full", functional="pzsic")
    else:
        solver = etdm.ETDM(d, precision=case["precision"])
    if kind in ("crystal", "sic"):
        C0, f = _full_reference(d, kind)
        solver.set_reference(torch.stack([c.to(torch.complex128) for c in C0]).cpu().numpy(), f)
    host = host.reshape(solver.var_shape)
    state = dict(case=case, solver=solver, a=torch.tensor(host, device=DEV))
    if kind == "minimize":
        state["x"] = torch.empty_like(state["a"])
    elif kind == "point":
        state["host"] = host
        state["fn"] = etdm.energy_function()
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "direction":
        return etdm.lbfgs_direction_noalloc(state["g"], state["S"], state["Y"], state["h0"],
                                            out=state["p"])
    solver = state["solver"]
    if kind == "minimize":  # from the start point, with an empty L-BFGS memory
        state["x"].copy_(state["a"])
        solver.lbfgs_reset()
        E, alpha, trials = solver.minimize(state["x"], case["steps"])
        return dict(E=E, alpha=alpha, trials=trials, a=state["x"])
    entry = case.get("entry", "device")
    if entry == "host":
        E, g = solver.energy_grad_host(state["host"])
    elif entry == "autograd":
        a = state["a"].detach().requires_grad_(True)
        E = state["fn"].apply(a, solver)
        (g,) = torch.autograd.grad(E, a)
        E = E.detach()
    else:
        E, g = solver.energy_grad(state["a"])
    return dict(E=E, g=g)


# ---- the least work -------------------------------------------------------------

def work(case):
    """Inputs read and outputs written once (variables, reference orbitals, T, the
    external potential), and the multiply-adds of the pairs of functions that
    overlap a grid point (each symmetric pair once, density and potential
    matrix), of the FFTs and of the products of the dense chains."""
    kind = case["kind"]
    if kind == "direction":
        n, m = case["n"], case["pairs"]
        return dict(bytes=8 * n * (2 * m + 3), flops=n * (8 * m + 2))
    by, fl = 0.0, 0.0
    for d in _systems(case):
        M, N, V = _sizes(d)
        G = float(np.prod(d["grid"]))
        reach = float((4.0 / 3.0 * math.pi * d["bf_rcut"] ** 3).sum() / np.prod(d["box"]))
        pairs = G * min(reach, 8.0 * M) ** 2
        fft = 2 * 2.5 * G * math.log2(G)
        if kind in ("crystal", "sic"):
            nk = len(_bloch(d, kind)[1])
            products = 4 if case.get("expm") == "ss" else 8
            by += nk * (16 * 2 * M * M + 8 * 2 * M * M) + 8 * G
            fl += 2 * pairs + fft + nk * products * 8.0 * M ** 3
            if kind == "sic":
                fl += N * (2 * pairs + fft)
        else:
            by += 8 * (2 * N * V + 2 * M * M + G)
            fl += 2 * pairs + fft + 8.0 * M * M * N + 6.0 * N * N * V + 20.0 * N ** 3
    if kind == "minimize":
        by, fl = by * (case["steps"] + 1), fl * (case["steps"] + 1)
    return dict(bytes=int(by), flops=int(fl))


# ---- the model in 64 bits ---------------------------------------------------------

def _t(x):
    return torch.tensor(np.asarray(x), dtype=F64, device=DEV)


def _images(d, reach):
    nm = [int(math.floor(reach / L)) + 1 for L in d["box"]]
    return itertools.product(*[range(-m, m + 1) for m in nm])


def _overlap_kinetic(d, k):
    """Analytic S(k) and T(k), images within r_c,mu + r_c,nu (real at the Gamma point)."""
    c = _t(d["pos"][d["bf_atom"]])
    al, rc = _t(d["bf_exp"]), _t(d["bf_rcut"])
    a, b = al[:, None], al[None, :]
    xi = a * b / (a + b)
    pre = (2.0 * (a * b).sqrt() / (a + b)) ** 1.5
    cut = (rc[:, None] + rc[None, :]) ** 2
    diff = c[:, None, :] - c[None, :, :]
    gamma = not np.any(k)
    S = torch.zeros_like(xi, dtype=F64 if gamma else torch.complex128)
    T = torch.zeros_like(S)
    for n in _images(d, 2.0 * float(d["bf_rcut"].max())):
        R2 = ((diff - _t(np.array(n) * d["box"])) ** 2).sum(-1)
        s = torch.where(R2 < cut, pre * torch.exp(-xi * R2), torch.zeros_like(xi))
        ph = 1.0 if gamma else complex(np.exp(2j * math.pi * float(np.dot(k, n))))
        S += ph * s
        T += ph * (xi * (3.0 - 2.0 * xi * R2) * s)
    return S, T


def _basis(d, k):
    """chi_mu,k on every grid point, (G, M)."""
    gamma = not np.any(k)
    nx, ny, nz = (int(v) for v in d["grid"])
    M = len(d["bf_exp"])
    al, rc2 = _t(d["bf_exp"]), _t(d["bf_rcut"]) ** 2
    norm = (2.0 * al / math.pi) ** 0.75
    c = _t(d["pos"][d["bf_atom"]])
    axes = [torch.arange(m, dtype=F64, device=DEV) * (float(L) / m)
            for m, L in zip((nx, ny, nz), d["box"])]
    X = torch.zeros((nx, ny * nz, M), dtype=F64 if gamma else torch.complex128, device=DEV)
    rmax = float(d["bf_rcut"].max())
    for n in _images(d, rmax):
        sq = [(ax[:, None] - (c[:, i] + n[i] * float(d["box"][i]))[None, :]) ** 2
              for i, ax in enumerate(axes)]
        yz = (sq[1][:, None, :] + sq[2][None, :, :]).reshape(ny * nz, M)
        ph = 1.0 if gamma else complex(np.exp(2j * math.pi * float(np.dot(k, n))))
        near = (sq[0] < rmax * rmax).any(1).cpu().numpy()
        for i in range(nx):
            if not near[i]:
                continue
            r2 = sq[0][i][None, :] + yz
            X[i] += ph * torch.where(r2 < rc2, norm * torch.exp(-al * r2), torch.zeros_like(r2))
    return X.reshape(nx * ny * nz, M)


class _Grid:
    """Potential and energy of a density on the grid."""

    def __init__(self, d):
        self.shape = tuple(int(v) for v in d["grid"])
        G = int(np.prod(self.shape))
        vol = float(np.prod(d["box"]))
        self.dV = vol / G
        g = [2.0 * math.pi * torch.fft.fftfreq(n, d=float(L) / n, dtype=F64, device=DEV)
             for n, L in zip(self.shape, d["box"])]
        G2 = (g[0] ** 2)[:, None, None] + (g[1] ** 2)[None, :, None] + (g[2] ** 2)[None, None, :]
        self.kernel = torch.where(G2 > 0, 4.0 * math.pi / G2, torch.zeros_like(G2))
        pos, Z = _t(d["pos"]), _t(d["Z"])
        ph = [torch.exp(-1j * g[i][:, None] * pos[None, :, i]) for i in range(3)]
        xy = (ph[0][:, None, :] * ph[1][None, :, :] * Z).reshape(-1, len(Z))
        ions = (xy @ ph[2].T).reshape(self.shape)
        vg = -self.kernel / vol * torch.exp(-0.5 * G2 * float(d["ion_sigma"]) ** 2) * ions
        self.vext = (torch.fft.ifftn(vg) * G).real.reshape(-1)

    def hartree(self, rho):
        return torch.fft.ifftn(torch.fft.fftn(rho.reshape(self.shape))
                               * self.kernel).real.reshape(-1)

    def energy_potential(self, rho):
        vh = self.hartree(rho)
        r = rho.clamp_min(0.0)
        cx = (3.0 / math.pi) ** (1.0 / 3.0)
        r13 = r ** (1.0 / 3.0)
        E = self.dV * (rho @ self.vext + 0.5 * (rho @ vh) - 0.75 * cx * (r @ r13))
        return E, self.vext + vh - cx * r13


def _density(X, C, f):
    phi = X @ C
    return ((phi.real ** 2 + phi.imag ** 2) if phi.is_complex() else phi * phi) @ f


def _exact_point(d, a):
    M, N, V = _sizes(d)
    k0 = np.zeros(3)
    S, T = _overlap_kinetic(d, k0)
    X, grid = _basis(d, k0), _Grid(d)
    w, Q = torch.linalg.eigh(S)
    half = (Q / w.sqrt()) @ Q.T
    hcore = T + grid.dV * (X.T @ (grid.vext[:, None] * X))
    order = np.argsort(torch.einsum("mj,mn,nj->j", half, hcore, half).cpu().numpy(),
                       kind="stable")
    C0 = half[:, torch.tensor(order, device=DEV)]
    A = _t(a).reshape(N, V).requires_grad_(True)
    full = torch.cat([torch.cat([A.new_zeros(N, N), A], 1),
                      torch.cat([-A.T, A.new_zeros(V, V)], 1)], 0)
    O = C0 @ torch.matrix_exp(full)[:, :N]
    f = torch.full((N,), 2.0, dtype=F64, device=DEV)
    with torch.no_grad():
        Egrid, v = grid.energy_potential(_density(X, O, f))
        H = grid.dV * (X.T @ (v[:, None] * X))
    kin = 2.0 * (O * (T @ O)).sum()
    lin = 2.0 * (O * (H @ O)).sum()  # its derivative is the grid energy's
    (g,) = torch.autograd.grad(kin + lin, A)
    return (kin + Egrid).detach(), g


def _exact_full(d, kind, expm, a):
    kpts, kw = _bloch(d, kind)
    M, N, _ = _sizes(d)
    C0, occ = _full_reference(d, kind)
    grid = _Grid(d)
    iu, iud = torch.triu_indices(M, M, 1, device=DEV), torch.triu_indices(M, M, 0, device=DEV)
    var, orbs = [], []
    rho = torch.zeros(grid.vext.numel(), dtype=F64, device=DEV)
    for k in range(len(kw)):
        x = _t(a[k * M * M:(k + 1) * M * M]).requires_grad_(True)
        re = torch.zeros((M, M), dtype=F64, device=DEV).index_put((iu[0], iu[1]), x[:len(iu[0])])
        im = torch.zeros((M, M), dtype=F64, device=DEV).index_put((iud[0], iud[1]),
                                                                  x[len(iu[0]):])
        A = torch.complex(re - re.T, im + im.T - torch.diag(torch.diagonal(im)))
        if expm == "ss":  # the gradient of Eq. 42: at exp(A) as the reference
            U = torch.matrix_exp(A.detach()) @ (torch.eye(M, device=DEV) + A - A.detach())
        else:
            U = torch.matrix_exp(A)
        n = int(np.count_nonzero(occ[k]))
        f = _t(occ[k][:n])
        C = (C0[k].to(torch.complex128) @ U)[:, :n]
        with torch.no_grad():
            rho += _density(_basis(d, kpts[k]).to(torch.complex128), C, f)
        var.append(x)
        orbs.append((C, f))
    E, v = grid.energy_potential(rho)
    g = []
    for k, (C, f) in enumerate(orbs):
        X = _basis(d, kpts[k]).to(torch.complex128)
        T = _overlap_kinetic(d, kpts[k])[1].to(torch.complex128)
        H = grid.dV * (X.conj().T @ (v[:, None] * X))
        kin = ((C.conj() * (T @ C)).real @ f).sum()
        lin = ((C.conj() * (H @ C)).real @ f).sum()
        E = E + kin.detach()
        if kind == "sic":  # - sum f (E_H[n] + E_x[n, 0]) over the unit orbital densities
            n = (X @ C).abs() ** 2
            cx = (6.0 / math.pi) ** (1.0 / 3.0)
            for i in range(n.shape[1]):
                e = grid.dV * (0.5 * (n[:, i] @ grid.hartree(n[:, i]))
                               - 0.75 * cx * (n[:, i].clamp_min(1e-300) ** (4.0 / 3.0)).sum())
                lin = lin - f[i] * e
                E = E - f[i] * e.detach()
        g.append(torch.autograd.grad(kin + lin, var[k])[0])
    return E, torch.cat(g)


def exact(case, seed):
    kind = case["kind"]
    if kind == "direction":
        s = prepare(case, seed)
        q = s["g"].clone()
        al = []
        for si, yi in zip(s["S"].flip(0), s["Y"].flip(0)):
            al.append((si @ q) / (si @ yi))
            q -= al[-1] * yi
        q = s["h0"] * q
        for si, yi, ai in zip(s["S"], s["Y"], reversed(al)):
            q += (ai - (yi @ q) / (si @ yi)) * si
        return -q
    # a minimization has no closed answer; the largest box would take minutes
    if kind == "minimize":
        return None
    systems = _systems(case)
    a = _variables(case, systems, seed)
    if kind in ("crystal", "sic"):
        E, g = _exact_full(systems[0], kind, case.get("expm", "eig"), a)
        return dict(E=E.reshape(1), g=g)
    if sum(float(np.prod(d["grid"])) * len(d["bf_exp"]) ** 2 for d in systems) > 4e11:
        return None
    parts, at = [], 0
    for d in systems:
        M, N, V = _sizes(d)
        parts.append(_exact_point(d, a[at:at + N * V]))
        at += N * V
    E = torch.stack([p[0] for p in parts])
    if kind == "batch":
        return dict(E=E, g=torch.cat([p[1].reshape(-1) for p in parts]))
    entry = case["entry"]
    g = parts[0][1]
    if entry == "host":
        return dict(E=float(E[0]), g=g.cpu().numpy())
    return dict(E=E[0] if entry == "autograd" else E, g=g)
