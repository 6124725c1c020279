"""Set-up in memory that holds a handle but not the tables of its faster passes."""
import numpy as np
import pytest

import etdm_synth as synth

pytestmark = pytest.mark.gpu


def launches(s, a, C0=None):
    """E, g and the kernel launches of a call (full A: from the orbitals C0, the
    phases of the reference's own being arbitrary)."""
    import torch
    if C0 is not None:
        s.set_reference(C0)
    s.set_profiling(True)
    s.stage_times()
    E, g = s.energy_grad(a)
    torch.cuda.synchronize()
    s.check()
    return float(E.item()), g, s.stage_times()[2]


@pytest.mark.parametrize("path", ["occvirt", "gamma", "k-points"])
def test_setup_without_room_for_the_tables(path):
    """Of the memory that a handle takes, its tables of X on the grid are optional
    (and the workspace of the large products).  With room for the rest, a set-up
    succeeds, as it did before there were tables, on the other kernels, with the
    same results to their rounding."""
    import torch
    from paper_2101_12597_gb300.etdm import ETDM
    if path == "occvirt":  # tables of some 170 MB, most of the handle
        d = synth.water_box(lattice=(3, 2, 2), box_ang=7.4, grid=(56, 56, 56), rcut_ang=3.5)
    elif path == "gamma":
        d = synth.crystal(cells=(3, 3, 3), spacing_ang=2.6, n_exp=3, Z=2.0, rcut_ang=3.0,
                          grid=(72, 72, 72), kmesh=1, kT_ev=0.5, a_sigma=0.02, seed=12)
    else:  # tables of some 500 MB, a quarter of the handle
        d = synth.crystal(cells=(4, 4, 8), spacing_ang=2.8, n_exp=4, Z=4.0, rcut_ang=4.0,
                          grid=(56, 56, 112), kmesh=2, kT_ev=0.5, a_sigma=0.01, seed=4)
    a = torch.tensor(d["a0"], dtype=torch.float64, device="cuda")

    def free():
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        return torch.cuda.mem_get_info()[0]

    ETDM(d).close()  # (loads what a first set-up loads)
    before = free()
    s = ETDM(d)
    takes = before - free()
    C0 = None
    if path != "occvirt":
        w, Q = np.linalg.eigh(s.get_array("S_k").reshape(-1, s.M, s.M))
        C0 = (Q / np.sqrt(w)[:, None, :]) @ Q.conj().transpose(0, 2, 1)
    E0, g0, n0 = launches(s, a, C0)
    s.close()
    leave = takes - ((200 << 20) if path == "k-points" else (12 << 20))
    fill = torch.empty(free() - leave, dtype=torch.uint8, device="cuda")
    try:
        s = ETDM(d)
        E1, g1, n1 = launches(s, a, C0)
        s.close()
    finally:
        del fill
        torch.cuda.empty_cache()
    dg = (g1 - g0).abs().max().item() / g0.abs().max().item()
    print(f"{path}: {takes >> 20} MB, launches {n0} -> {n1}, dE={abs(E1 - E0):.1e} dg={dg:.1e}")
    assert n1 < n0  # the passes on tables take more launches
    assert abs(E1 - E0) < 1e-9 and dg <= 1e-9


def test_batch_without_room_for_every_table():
    """An FP64 batch whose members fit without their tables: those of the first
    members are given back when a later one has no room."""
    import torch
    from paper_2101_12597_gb300.etdm import ETDMBatch
    systems = [synth.water_box(lattice=(3, 2, 2), box_ang=7.4, grid=(56, 56, 56), rcut_ang=3.5, seed=i)
               for i in range(8)]
    a = torch.tensor(np.concatenate([d["a0"].ravel() for d in systems]), device="cuda")

    def free():
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        return torch.cuda.mem_get_info()[0]

    ETDMBatch(systems[:1], precision="fp64").close()
    before = free()
    b = ETDMBatch(systems, precision="fp64")
    takes = before - free()
    E0, g0 = (x.clone() for x in b.energy_grad(a))
    torch.cuda.synchronize()
    b.close()
    # room for three members with their tables and part of a fourth's memory
    leave = int(3.2 * takes / len(systems))
    fill = torch.empty(free() - leave, dtype=torch.uint8, device="cuda")
    try:
        b = ETDMBatch(systems, precision="fp64")
        E1, g1 = (x.clone() for x in b.energy_grad(a))
        torch.cuda.synchronize()
        b.close()
    finally:
        del fill
        torch.cuda.empty_cache()
    print(f"{takes >> 20} MB, {leave >> 20} left: dE={(E1 - E0).abs().max().item():.1e}")
    assert (E1 - E0).abs().max().item() < 1e-9
    assert (g1 - g0).abs().max().item() <= 1e-9 * g0.abs().max().item()
