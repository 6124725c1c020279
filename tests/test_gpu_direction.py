"""The allocation-free direction where its work vector changes place: within
the registers (one and many blocks), the first and a partly filled
shared-memory slot, and beyond the on-chip capacity of a block per SM."""
import numpy as np
import pytest

import etdm_synth as synth

pytestmark = pytest.mark.gpu

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


THREADS, REGS, SLOTS = 512, 16, 55


@pytest.mark.parametrize("m", [0, 1, 4])
@pytest.mark.parametrize("where", ["one", "regs", "slot", "partial", "memory"])
def test_direction_over_the_storage_ranges(where, m):
    """Tolerance: each of the 2m dot products and updates rounds at 2^-53 of its
    terms; n terms of one sign at most, so n 2^-53 (6e-10 at the largest n) of
    the largest entry bounds a dot product's error; 1e-9 of max|p|."""
    import torch
    from paper_2101_12597_gb300 import etdm
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    row = sms * THREADS  # elements of one register or slot over the grid
    n = {"one": 3, "regs": REGS * row, "slot": REGS * row + 1, "partial": (REGS + 3) * row - 77,
         "memory": (REGS + SLOTS) * row + 1234}[where]
    if where == "memory" and m == 4:
        pytest.skip("the oracle's copies would take 3 GB")
    g = synth.direction(n, 1)
    h0 = 0.5 + np.abs(synth.direction(n, 2))
    S = synth.direction((m, n), 3, 0.1) if m else np.zeros((0, n))
    Y = S * (0.5 + np.abs(synth.direction((1, n), 4))) if m else np.zeros((0, n))
    dev = lambda x: torch.tensor(x, dtype=torch.float64, device="cuda")
    p = etdm.lbfgs_direction_noalloc(dev(g), dev(S) if m else None, dev(Y) if m else None, dev(h0))
    etdm.lbfgs_direction_noalloc_status()
    want = two_loop(g, S, Y, h0)
    assert np.abs(p.cpu().numpy() - want).max() <= 1e-9 * np.abs(want).max()
