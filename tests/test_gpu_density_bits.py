"""The FP64 density and potential matrix where the functions are small: every
value of a function on the grid keeps FP64's 53 bits, in its tail too, so rho
is exact relative to its own terms in the vacuum around a molecule, where
single functions of 1e-8 to 1e-14 of their peak make it up."""
import numpy as np
import pytest

import etdm_synth as synth
from oracle.etdm_kpoints import BlochOracle
from oracle.etdm_oracle import Oracle

pytestmark = pytest.mark.gpu


def molecule(exps):
    """Six atoms within 4 A in the middle of a 12 A box."""
    d = synth.random_atoms(n_atoms=6, box_ang=4.0, grid=(30, 32, 36), exps=exps, a_sigma=0.05, seed=3)
    A = synth.ANGSTROM
    d["box"] = np.full(3, 12.0 * A)
    d["pos"] = np.asarray(d["pos"]) + 4.0 * A
    return d


def relative_error(rho, X, D):
    """Largest error of rho_p over sum_ab |X_pa D_ab X_pb| (points that it is not
    below 1e-250 at: FP64's own range)."""
    ref = ((X @ D) * X.conj()).sum(1).real
    mag = ((np.abs(X) @ np.abs(D)) * np.abs(X)).sum(1)
    at = mag > 1e-250
    assert at.sum() > 1000 and mag[at].min() < 1e-20 * mag.max()  # the vacuum is there
    return (np.abs(rho.reshape(-1) - ref)[at] / mag[at]).max()


# A value of X carries the roundings of alpha dx^2 (dx = grid point minus centre
# and image: 3 roundings of the box length L, 2 alpha dx dL each) and of three
# exponentials, both sides alike: with alpha <= 4, dx <= 10, L = 23 bohr at most
# 3 x 3 x 2 x 4 x 10 x 23 x 2^-53 < 2e-12; two values per term, two sides, and
# far smaller sums: 1e-11.
TOL = 1e-11


@pytest.mark.parametrize("exps", [(0.5, 1.5), (0.25, 4.0)])
def test_density_relative_to_its_terms(exps):
    import torch
    from paper_2101_12597_gb300.etdm import ETDM
    d = molecule(exps)
    o, s = Oracle(d), ETDM(d)
    s.energy_grad(torch.tensor(d["a0"], dtype=torch.float64, device="cuda"))
    torch.cuda.synchronize()
    s.check()
    D = s.get_array("D").reshape(o.M, o.M)
    err = relative_error(s.get_array("rho"), o.X(), D)
    print(f"{exps}: {err:.1e}")
    assert err <= TOL
    # H - T against X^T v X: the largest element of a row and of a column set
    # the scale of what FP64 sums keep (n_points roundings at most)
    V = s.get_array("H").reshape(o.M, o.M) - s.get_array("T").reshape(o.M, o.M)
    X, v = o.X(), s.get_array("vtot").reshape(-1)
    ref = o.dV * (X.T @ (v[:, None] * X))
    size = np.sqrt(np.outer(np.diag(o.dV * (X.T @ (np.abs(v)[:, None] * X))),
                            np.diag(o.dV * (X.T @ (np.abs(v)[:, None] * X)))))
    T = np.abs(s.get_array("T").reshape(o.M, o.M))
    assert (np.abs(V - ref) <= TOL * size + 4 * 2.0 ** -52 * (T + size)).all()
    s.close()


@pytest.mark.parametrize("kmesh", [1, 2])
def test_crystal_density_relative_to_its_terms(kmesh):
    """The full-A path: images merged at the Gamma point, an entry per image with
    k-points (two atoms in a long cell)."""
    import torch
    from paper_2101_12597_gb300.etdm import ETDM
    d = synth.crystal(cells=(1, 1, 2), spacing_ang=6.0, jitter_ang=0.1, exps=(0.5, 1.5), Z=1.0,
                      rcut_ang=5.9, grid=(16, 15, 32), kmesh=kmesh, kT_ev=0.5, a_sigma=0.05, seed=6)
    bo = BlochOracle(d)
    s = ETDM(d)
    s.energy_grad(torch.tensor(d["a0"], dtype=torch.float64, device="cuda"))
    torch.cuda.synchronize()
    s.check()
    D = s.get_array("D_k").reshape(bo.nk, bo.M, bo.M)
    rho = s.get_array("rho").reshape(-1)
    ref, mag = np.zeros(bo.G), np.zeros(bo.G)
    for k in range(bo.nk):
        X = bo.Xk(k)
        ref += ((X @ D[k]) * X.conj()).sum(1).real
        mag += ((np.abs(X) @ np.abs(D[k])) * np.abs(X)).sum(1)
    err = (np.abs(rho - ref) / mag).max()
    print(f"kmesh={kmesh}: {err:.1e}, smallest {mag.min() / mag.max():.1e}")
    assert mag.min() < 1e-6 * mag.max() and err <= TOL
    s.close()


@pytest.mark.parametrize("exps", [(2.0, 8.0), (0.8, 3.0)])
def test_potential_over_atoms_without_electrons(exps):
    """Half of a row of atoms holds no electron, and A = 0, so the density there is
    of the tails of the others' orbitals (1e-8 to 1e-40 of the largest), in tiles
    that also list occupied functions.  rho^(1/3) passes its relative error on:
    rho to 1e-11 of its terms as above, H to 64 roundings of its largest element
    (v to a few roundings times the sums over points)."""
    import torch
    from paper_2101_12597_gb300.etdm import ETDM
    d = synth.crystal(cells=(2, 2, 12), spacing_ang=2.6, Z=2.0, rcut_ang=3.0, kT_ev=0.5, a_sigma=0.05,
                      seed=12, exps=exps, grid=(14, 14, 84), kmesh=2)
    bo = BlochOracle(d)
    C0 = bo.lowdin_reference()
    f = np.zeros(bo.M)
    f[:bo.M // 2:2] = 1.0  # an orbital of each atom of the first half
    f *= bo.N / f.sum()
    occ = [2.0 * w * f for w in bo.kw]
    bo.reference_k()
    bo.set_reference(C0, occ)
    s = ETDM(d)
    s.set_reference(np.array(C0), np.array(occ))
    a = np.zeros(bo.nk * bo.nvar)
    E, g = s.energy_grad(torch.tensor(a, dtype=torch.float64, device="cuda"))
    torch.cuda.synchronize()
    s.check()
    E_ref, g_ref, ex = bo.energy_grad(a, want=True)
    D = s.get_array("D_k").reshape(bo.nk, bo.M, bo.M)
    H = s.get_array("H_k").reshape(bo.nk, bo.M, bo.M)
    ref, mag, dH, big = np.zeros(bo.G), np.zeros(bo.G), 0.0, 0.0
    for k in range(bo.nk):
        X = bo.Xk(k)
        ref += ((X @ D[k]) * X.conj()).sum(1).real
        mag += ((np.abs(X) @ np.abs(D[k])) * np.abs(X)).sum(1)
        dH = max(dH, np.abs(H[k] - ex["k"][k]["H"]).max())
        big = max(big, np.abs(ex["k"][k]["H"]).max())
    err = (np.abs(s.get_array("rho").reshape(-1) - ref) / mag).max()
    print(f"{exps}: rho {err:.1e}, H {dH:.1e} of {big:.1e}, smallest rho {mag.min():.1e}")
    assert err <= TOL and dH <= 64 * 2.0 ** -53 * big
    assert abs(float(E.item()) - E_ref) < 1e-9
    s.close()
