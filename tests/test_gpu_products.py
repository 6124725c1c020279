"""The full-A path's complex products at the sizes where their kernels can go
wrong, through E and the gradient against the k-point oracle: FP64 tiles with
a remainder and one k-point (20), the largest on the FP64 kernel (64), tensor
cores with a K tail and a partial column tile (80), a second block of 128 rows
(144); the eigensolver's panels of 16 columns from the first size that takes
them, whole (128) and with a remainder of 7 (135), for eight matrices and for
one, whose blocks hold a few rows each; with exp(A) by both routes."""
import numpy as np
import pytest

import etdm_synth as synth
from oracle.etdm_kpoints import BlochOracle

pytestmark = pytest.mark.gpu

SYSTEMS = {
    20: dict(cells=(2, 1, 2), n_exp=5, grid=(16, 15, 14), kmesh=1),
    64: dict(cells=(2, 2, 2), n_exp=8, grid=(16, 15, 14), kmesh=2),
    80: dict(cells=(2, 5, 2), n_exp=4, grid=(14, 24, 15), kmesh=2),
    144: dict(cells=(3, 3, 4), n_exp=4, grid=(20, 18, 24), kmesh=2),
    128: dict(cells=(4, 2, 4), n_exp=4, grid=(24, 15, 24), kmesh=1),
    135: dict(cells=(3, 3, 5), n_exp=3, grid=(20, 18, 28), kmesh=2),
}


@pytest.mark.parametrize("expm", ["eig", "ss"])
@pytest.mark.parametrize("M", list(SYSTEMS))
def test_energy_gradient_over_product_sizes(M, expm):
    """Loewdin reference and occupations with a partly filled edge handed to
    both sides.  Tolerances: those of the path's other parity tests (1e-9 Ha,
    1e-9 of max|g|)."""
    import torch
    from paper_2101_12597_gb300.etdm import ETDM
    kw = dict(SYSTEMS[M])
    exps = [0.3 * 40.0 ** (e / (kw["n_exp"] - 1)) for e in range(kw["n_exp"])]
    d = synth.crystal(spacing_ang=2.6, Z=2.0, rcut_ang=3.0, kT_ev=0.5, a_sigma=0.05, seed=12,
                      exps=exps, **kw)
    bo = BlochOracle(d)
    assert bo.M == M
    f = 1.0 / (1.0 + np.exp((np.arange(M) - bo.N + 0.5) / 2.0))
    f *= bo.N / f.sum()
    occ = [2.0 * w * f for w in bo.kw]
    C0 = bo.lowdin_reference()
    bo.reference_k()
    bo.set_reference(C0, occ)
    s = ETDM(d, expm=expm)
    s.set_reference(np.array(C0), np.array(occ))
    E, g = s.energy_grad(torch.tensor(d["a0"], dtype=torch.float64, device="cuda"))
    torch.cuda.synchronize()
    s.check()
    E_ref, g_ref = bo.energy_grad(d["a0"]) if expm == "eig" else bo.energy_grad_approx(d["a0"])
    dE = abs(float(E.item()) - E_ref)
    dg = np.abs(g.cpu().numpy() - g_ref).max() / np.abs(g_ref).max()
    print(f"M={M} {expm}: |dE|={dE:.2e} max|dg|/max|g|={dg:.2e}")
    assert dE < 1e-9 and dg <= 1e-9
    s.close()
