"""The dense chains kept in shared memory (M <= 32), at the ends of their range:
two functions, odd sizes, one and two 16-wide K chunks, more outputs than
threads, N above and below V, matrices beyond the shared memory (the general
chains), with no and with several doublings."""
import numpy as np
import pytest

import etdm_synth as synth
from oracle.etdm_oracle import Oracle

pytestmark = pytest.mark.gpu

SIZES = {  # (M, N): atoms, exponents, Z
    (2, 1): (2, (1.0,), 1.0),
    (15, 5): (5, (0.6, 1.5, 4.0), 2.0),
    (30, 20): (10, (0.6, 1.5, 4.0), 4.0),
    (32, 8): (16, (0.7, 2.0), 1.0),
    (32, 16): (16, (0.7, 2.0), 2.0),
    (32, 28): (8, (0.6, 1.2, 2.4, 4.8), 7.0),
}


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("spread", [0.03, 0.6])
@pytest.mark.parametrize("size", list(SIZES))
def test_energy_gradient_over_small_sizes(size, spread, precision):
    """Tolerances: those of the two paths' other parity tests (1e-9 Ha and 1e-9
    of max|g|; 1e-6 Ha and 1e-5 of max|g|)."""
    import torch
    from paper_2101_12597_gb300.etdm import ETDM
    n, exps, Z = SIZES[size]
    d = synth.random_atoms(n_atoms=n, exps=exps, Z=Z, rcut_ang=2.8, grid=(30, 28, 33), a_sigma=spread,
                           seed=31)
    o, s = Oracle(d), ETDM(d, precision=precision)
    assert (len(d["bf_exp"]), d["n_electrons"] // 2) == size
    a = torch.tensor(d["a0"], dtype=torch.float64, device="cuda")
    E, g = s.energy_grad(a)
    torch.cuda.synchronize()
    s.check()
    E_ref, g_ref = o.energy_grad(d["a0"])
    dE = abs(float(E.item()) - E_ref)
    dg = np.abs(g.cpu().numpy() - g_ref).max() / np.abs(g_ref).max()
    print(f"{size} {spread} {precision}: |dE|={dE:.2e} max|dg|/max|g|={dg:.2e}")
    assert dE < (1e-9 if precision == "fp64" else 1e-6)
    assert dg <= (1e-9 if precision == "fp64" else 1e-5)
    s.close()
