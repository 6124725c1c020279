"""Non-finite density matrices on the FP64 grid passes, which hold numbers in fixed
point."""
import numpy as np
import pytest

import etdm_synth as synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("kmesh", [1, 2])
def test_density_of_a_non_finite_density_matrix(kmesh, bad):
    """A non-finite D reaches rho as one (it is no fixed-point number), and the
    call reports the numeric error."""
    import torch
    from paper_2101_12597_gb300.etdm import ETDM, EtdmError
    d = synth.tiny_crystal(rcut_ang=3.0, kmesh=kmesh)
    s = ETDM(d)
    a = np.array(d["a0"])
    E, _ = s.energy_grad(torch.tensor(a, dtype=torch.float64, device="cuda"))
    torch.cuda.synchronize()
    s.check()
    assert np.isfinite(s.get_array("rho")).all()
    a[1] = bad
    E, _ = s.energy_grad(torch.tensor(a, dtype=torch.float64, device="cuda"))
    torch.cuda.synchronize()
    assert not np.isfinite(float(E.item()))
    rho = s.get_array("rho")
    assert not np.isfinite(s.get_array("D_k")).all()
    assert not np.isfinite(rho).any()  # every tile lists every function of this cell
    with pytest.raises(EtdmError):
        s.check()
    s.close()
