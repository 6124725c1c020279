"""Which kernels run, by the launches of a call, and the results of the ones that
few systems take: FP64 grid passes on tables (a density in 2 launches, a
potential matrix in 4) up to 128 functions or images per tile, else one launch
each; full-A products on the tensor cores (3 launches a product) from M = 80 on
with 8 k-points."""
import numpy as np
import pytest

import etdm_synth as synth
from oracle.etdm_oracle import Oracle

pytestmark = pytest.mark.gpu

# dense chains 2, potential 5; with the tables 6 more, without 2
TABLES, PLAIN = 13, 9
# iA and phases 2, eigensolver 7, other steps 13, products 9; tables or not
K_TABLES, K_PLAIN = 2 + 7 + 13 + 9 + 6, 2 + 7 + 13 + 9 + 2
# products on the tensor cores: 3 launches each, U - I one
K_OZ = K_TABLES + 2 * 9 + 1


def evaluate(d, **kw):
    import torch
    from paper_2101_12597_gb300.etdm import ETDM
    s = ETDM(d, **kw)
    s.set_profiling(True)
    s.stage_times()
    E, g = s.energy_grad(torch.tensor(d["a0"], dtype=torch.float64, device="cuda"))
    torch.cuda.synchronize()
    s.check()
    out = float(E.item()), g.cpu().numpy(), s.stage_times()[2]
    s.close()
    return out


@pytest.mark.parametrize("M,launches", [(16, TABLES), (66, TABLES), (128, TABLES), (140, PLAIN)])
def test_gamma_point_passes(M, launches):
    """Every function of 128 in every tile still takes the tables; of 140, some 134
    reach one tile.  Tolerances: those of the FP64 path's parity tests."""
    d = synth.random_atoms(n_atoms=M, exps=(2.0,), rcut_ang=3.6, grid=(30, 28, 33), a_sigma=0.02,
                           min_sep_ang=0.9, seed=21)
    E, g, n = evaluate(d)
    assert n == launches
    if launches == PLAIN:
        E_ref, g_ref = Oracle(d).energy_grad(d["a0"])
        print(f"M={M}: |dE|={abs(E - E_ref):.2e} dg {np.abs(g - g_ref).max() / np.abs(g_ref).max():.2e}")
        assert abs(E - E_ref) < 1e-9 and np.abs(g - g_ref).max() <= 1e-9 * np.abs(g_ref).max()


CRYSTALS = {
    "few images": (K_TABLES, dict(cells=(2, 1, 1), spacing_ang=2.2, exps=(0.6, 2.4), rcut_ang=2.4,
                                  grid=(24, 12, 12))),
    "88 images": (K_TABLES, dict(cells=(2, 1, 1), spacing_ang=2.2, exps=(0.6, 2.4), rcut_ang=4.2,
                                 grid=(24, 12, 12))),
    "over 128": (K_PLAIN, dict(cells=(2, 1, 1), spacing_ang=1.6, exps=(1.5, 6.0, 24.0), rcut_ang=3.1,
                               grid=(22, 12, 11))),
    "M = 64": (K_TABLES, dict(cells=(2, 4, 2), spacing_ang=2.6, exps=(0.3, 1.0, 3.5, 12.0), rcut_ang=3.0,
                              grid=(14, 24, 14))),
    "M = 80": (K_OZ, dict(cells=(2, 5, 2), spacing_ang=2.6, exps=(0.3, 1.0, 3.5, 12.0), rcut_ang=3.0,
                          grid=(14, 24, 15))),
}


@pytest.mark.parametrize("which", list(CRYSTALS))
def test_full_A_kernels(which):
    launches, kw = CRYSTALS[which]
    d = synth.crystal(Z=1.0, kmesh=2, kT_ev=0.5, a_sigma=0.05, jitter_ang=0.1, seed=6, **kw)
    assert evaluate(d)[2] == launches


def two_loop(g, S, Y, h0):
    """p = -H g over the pairs oldest (0) to newest (Sec. 3.1)."""
    q, al = g.copy(), []
    for s, y in zip(S[::-1], Y[::-1]):
        al.append((s @ q) / (s @ y))
        q -= al[-1] * y
    q *= h0
    for s, y, a in zip(S, Y, al[::-1]):
        q += (a - (y @ q) / (s @ y)) * s
    return -q


@pytest.mark.parametrize("m", [2, 4])
def test_direction_of_several_pairs_beyond_the_chip(m):
    """A work vector that does not fit the registers and shared memory of every SM
    (71 elements a thread), with the updates between the pairs of both loops.
    Tolerance as for the other storage ranges: n 2^-53 (6e-10) of the largest entry
    per dot product; 1e-9."""
    import torch
    from paper_2101_12597_gb300 import etdm
    n = (16 + 55) * torch.cuda.get_device_properties(0).multi_processor_count * 512 + 1234
    g = synth.direction(n, 1)
    h0 = 0.5 + np.abs(synth.direction(n, 2))
    S = synth.direction((m, n), 3, 0.1)
    Y = S * (0.5 + np.abs(synth.direction((1, n), 4)))
    dev = lambda x: torch.tensor(x, dtype=torch.float64, device="cuda")
    p = etdm.lbfgs_direction_noalloc(dev(g), dev(S), dev(Y), dev(h0))
    etdm.lbfgs_direction_noalloc_status()
    want = two_loop(g, S, Y, h0)
    assert np.abs(p.cpu().numpy() - want).max() <= 1e-9 * np.abs(want).max()
