"""Density matrices of functions that hold little charge, on the products of the
tensor cores (M of 80 and more with 8 k-points), whose rows share a power of
two: with A = 0 the orbitals are the reference's, and D keeps its relative
accuracy over atoms without electrons (D of 1e-8 to 1e-20 of the largest)."""
import numpy as np
import pytest

import etdm_synth as synth
from oracle.etdm_kpoints import BlochOracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("expm", ["eig", "ss"])
@pytest.mark.parametrize("exps", [(2.0, 8.0), (0.8, 3.0)])
def test_density_matrix_relative_to_its_diagonal(exps, expm):
    """Each of the N terms of D_ab = sum_j f_j O_aj conj(O_bj) rounds three times at
    2^-53 of itself, and their moduli add up to (D_aa D_bb)^(1/2) at most: 2^-53
    times 3, the sums' log2 N or so, both sides: 32."""
    import torch
    from paper_2101_12597_gb300.etdm import ETDM
    d = synth.crystal(cells=(2, 2, 12), spacing_ang=2.6, Z=2.0, rcut_ang=3.0, kT_ev=0.5, a_sigma=0.05,
                      seed=12, exps=exps, grid=(14, 14, 84), kmesh=2)
    bo = BlochOracle(d)
    M, nk = bo.M, bo.nk
    C0 = np.array(bo.lowdin_reference())
    f = np.zeros(M)
    f[:M // 2:2] = 1.0  # an orbital of each atom of the first half, unequally filled
    f *= 1.0 + 0.3 * np.cos(np.arange(M))
    f *= bo.N / f.sum()
    occ = np.array([2.0 * w * f for w in bo.kw])
    s = ETDM(d, expm=expm)
    s.set_reference(C0, occ)
    a = torch.zeros(nk * M * M, dtype=torch.float64, device="cuda")
    s.energy_grad(a)
    torch.cuda.synchronize()
    s.check()
    D = s.get_array("D_k").reshape(nk, M, M)
    worst, least = 0.0, 1.0
    for k in range(nk):
        ref = (C0[k] * occ[k]) @ C0[k].conj().T
        q = np.sqrt(np.diag(ref).real)
        least = min(least, q.min() / q.max())
        worst = max(worst, (np.abs(D[k] - ref) / np.outer(q, q)).max())
    print(f"{exps} {expm}: {worst:.1e} (smallest D_aa^(1/2) {least:.1e})")
    assert least < 1e-3 and worst <= 32 * 2.0 ** -53
    s.close()
