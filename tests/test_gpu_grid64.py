"""The FP64 grid passes over the list lengths where their tensor-core kernels
change shape: nearly every function reaches every tile, so a tile has up to M
entries, in passes of 64 columns with a last one of 16, 32 or 64, on grids of
partial tiles, also at the reference, whose density leaves the unoccupied
functions' atoms nearly empty; and with k-points an entry per image up to and
beyond the 128 that the kernels take."""
import numpy as np
import pytest

import etdm_synth as synth
from oracle.etdm_kpoints import BlochOracle
from oracle.etdm_oracle import Oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("start", ["seeded", "reference"])
@pytest.mark.parametrize("M", [16, 18, 34, 64, 66, 82, 128])
def test_energy_gradient_over_list_lengths(M, start):
    """Tolerances: those of the FP64 path's other parity tests (1e-9 Ha, 1e-9 of
    max|g|); rho to 1e-11 of its largest value."""
    import torch
    from paper_2101_12597_gb300.etdm import ETDM
    d = synth.random_atoms(n_atoms=M, exps=(2.0,), rcut_ang=3.6, grid=(30, 28, 33), a_sigma=0.02,
                           min_sep_ang=0.9, seed=21)
    o, s = Oracle(d), ETDM(d)
    a = d["a0"] if start == "seeded" else np.zeros_like(d["a0"])
    E, g = s.energy_grad(torch.tensor(a, dtype=torch.float64, device="cuda"))
    torch.cuda.synchronize()
    s.check()
    E_ref, g_ref = o.energy_grad(a)
    rho = o.density(o.density_matrix(o.orbitals(a)))
    dE = abs(float(E.item()) - E_ref)
    dg = np.abs(g.cpu().numpy() - g_ref).max() / np.abs(g_ref).max()
    dr = np.abs(s.get_array("rho").reshape(rho.shape) - rho).max() / rho.max()
    print(f"M={M} {start}: |dE|={dE:.2e} max|dg|/max|g|={dg:.2e} rho {dr:.2e}")
    assert dE < 1e-9 and dg <= 1e-9 and dr <= 1e-11
    s.close()


CRYSTALS = {
    "few images": dict(cells=(2, 1, 1), spacing_ang=2.2, exps=(0.6, 2.4), rcut_ang=2.4, grid=(24, 12, 12)),
    "88 images": dict(cells=(2, 1, 1), spacing_ang=2.2, exps=(0.6, 2.4), rcut_ang=4.2, grid=(24, 12, 12)),
    "over 128": dict(cells=(2, 1, 1), spacing_ang=1.6, exps=(1.5, 6.0, 24.0), rcut_ang=3.1,
                     grid=(22, 12, 11)),
}


@pytest.mark.parametrize("which", list(CRYSTALS))
def test_crystal_over_image_counts(which):
    import torch
    from paper_2101_12597_gb300.etdm import ETDM
    d = synth.crystal(Z=1.0, kmesh=2, kT_ev=0.5, a_sigma=0.05, jitter_ang=0.1, seed=6, **CRYSTALS[which])
    bo = BlochOracle(d)
    C0 = bo.lowdin_reference()
    f = bo.reference_k()["f"]
    bo.set_reference(C0, f)
    s = ETDM(d)
    s.set_reference(np.array(C0), np.array(f))
    E, g = s.energy_grad(torch.tensor(d["a0"], dtype=torch.float64, device="cuda"))
    torch.cuda.synchronize()
    s.check()
    E_ref, g_ref = bo.energy_grad(d["a0"])
    assert abs(float(E.item()) - E_ref) < 1e-9
    assert np.abs(g.cpu().numpy() - g_ref).max() <= 1e-9 * np.abs(g_ref).max()
    s.close()
