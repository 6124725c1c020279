"""Handles of different sizes evaluated by host threads of their own."""
import threading

import pytest

import etdm_synth as synth

pytestmark = pytest.mark.gpu


def test_two_threads_with_different_grids():
    """Each thread evaluates its own FP64 system on its own stream; lines of 256
    points take more shared memory than a launch has by default, those of 16 much
    less.  Every call succeeds and repeats its energy."""
    import torch
    from paper_2101_12597_gb300.etdm import ETDM
    # (some 65 x 65 lines of 256 points: eight a block, 70 KB)
    long = synth.random_atoms(n_atoms=2, grid=(65, 66, 256), exps=(1.5,), rcut_ang=2.0, seed=5)
    short = synth.random_atoms(n_atoms=2, grid=(16, 16, 16), exps=(1.5,), rcut_ang=2.0, seed=5)
    solvers = [ETDM(d) for d in (long, short)]
    errors, energies = [], [set(), set()]

    def work(i, d, s):
        try:
            torch.cuda.set_device(0)
            stream = torch.cuda.Stream()
            a = torch.tensor(d["a0"], dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            for _ in range(400 if i else 100):
                E, g = s.energy_grad(a, stream=stream)
                stream.synchronize()
                energies[i].add(float(E.item()))
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    ts = [threading.Thread(target=work, args=(i, d, s))
          for i, (d, s) in enumerate(zip((long, short), solvers))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors
    assert all(len(e) == 1 for e in energies), energies
    for s in solvers:
        s.close()
