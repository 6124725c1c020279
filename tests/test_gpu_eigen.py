"""exp(A) and the Eq. 39 adjoint of A(k) with eigenvalues of very different
size: the null space of a calculation from A = 0 (its occupied-occupied and
virtual-virtual blocks stay zero where the occupations are equal), low rank,
and a part decoupled from the rest and far smaller; at sizes of each reduction
to tridiagonal form (one block, groups, panels; eight matrices and one)."""
import numpy as np
import pytest

import etdm_synth as synth
from oracle.etdm_kpoints import BlochOracle

pytestmark = pytest.mark.gpu

# M: atoms per edge, Gaussians per atom, grid, k-mesh
SYSTEMS = {
    64: dict(cells=(2, 4, 2), n_exp=4, grid=(14, 24, 14), kmesh=2),
    96: dict(cells=(2, 4, 3), n_exp=4, grid=(14, 24, 18), kmesh=2),
    144: dict(cells=(3, 3, 4), n_exp=4, grid=(20, 18, 24), kmesh=2),
    150: dict(cells=(5, 5, 2), n_exp=3, grid=(28, 28, 14), kmesh=1),
    256: dict(cells=(4, 4, 4), n_exp=4, grid=(24, 24, 24), kmesh=2),
    512: dict(cells=(4, 4, 8), n_exp=4, grid=(24, 24, 48), kmesh=2),
}
KINDS = [(64, "zero blocks"), (144, "zero blocks"), (150, "zero blocks"), (256, "zero blocks"),
         (512, "zero blocks"), (96, "rank 20"), (150, "rank 20"), (64, "decoupled 1e-13"),
         (64, "decoupled 1e-15"), (64, "decoupled 1e-16"), (144, "decoupled 1e-13"),
         (150, "decoupled 1e-16"), (144, "dense"), (150, "dense"), (64, "one pair"), (150, "one pair")]


def variables(kind, M, N, nk, seed):
    """Packed reals (Re a_ij, i < j; Im a_ij, i <= j) of every A(k)."""
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(nk):
        X = 0.05 * (rng.normal(size=(M, M)) + 1j * rng.normal(size=(M, M)))
        if kind == "rank 20":
            Y = rng.normal(size=(M, 20)) + 1j * rng.normal(size=(M, 20))
            X = 1j * (Y * (0.05 * rng.normal(size=20) / M)) @ Y.conj().T
        A = X - X.conj().T if kind != "rank 20" else X
        if kind == "zero blocks":
            A[:N, :N] = 0.0
            A[N:, N:] = 0.0
        elif kind.startswith("decoupled"):
            h = M // 2
            A[:h, h:] = 0.0
            A[h:, :h] = 0.0
            A[h:, h:] *= float(kind.split()[1])
        elif kind == "one pair":
            A[:] = 0.0
            A[3, M - 2], A[M - 2, 3] = 0.3, -0.3
        out += [A[np.triu_indices(M, 1)].real, A[np.triu_indices(M)].imag]
    return np.concatenate(out)


@pytest.mark.parametrize("M,kind", KINDS)
def test_exponential_and_adjoint(M, kind):
    """D(k) against C0 exp(A) f exp(A)^+ C0^+ and g against Eq. 39 of the device's
    own H(k), both with a dense eigendecomposition of iA(k) on the host.  Any
    backward stable route leaves some n 2^-52 in exp(A) (|A| of order one): 16 n
    2^-52, times the norms that follow it."""
    import torch
    from paper_2101_12597_gb300.etdm import ETDM
    kw = dict(SYSTEMS[M])
    nexp = kw["n_exp"]
    d = synth.crystal(spacing_ang=2.6, Z=2.0, rcut_ang=3.0, kT_ev=0.5, a_sigma=0.05, seed=12,
                      exps=[0.3 * 40.0 ** (e / (nexp - 1)) for e in range(nexp)], **kw)
    bo = BlochOracle(d)
    assert bo.M == M
    N, nk = bo.N, bo.nk
    s = ETDM(d)
    S = s.get_array("S_k").reshape(nk, M, M)
    C0 = []
    for k in range(nk):  # (any orthonormal orbitals)
        w, Q = np.linalg.eigh(0.5 * (S[k] + S[k].conj().T))
        C0.append((Q / np.sqrt(w)) @ Q.conj().T)
    occ = np.array([np.where(np.arange(M) < N, 2.0 * w, 0.0) for w in bo.kw])
    if kind == "dense":
        occ = np.array([2.0 * w * bo.N / (1.0 + np.exp((np.arange(M) - N) / 2.0))
                        / (1.0 / (1.0 + np.exp((np.arange(M) - N) / 2.0))).sum() for w in bo.kw])
    s.set_reference(np.array(C0), occ)
    a = variables(kind, M, N, nk, 5)
    E, g = s.energy_grad(torch.tensor(a, dtype=torch.float64, device="cuda"))
    torch.cuda.synchronize()
    s.check()
    H = s.get_array("H_k").reshape(nk, M, M)
    D = s.get_array("D_k").reshape(nk, M, M)
    g = g.cpu().numpy().reshape(nk, -1)
    worst = [0.0, 0.0]
    eps = 16 * M * 2.0 ** -52
    for k in range(nk):
        A = bo.A_of(a[k * M * M:(k + 1) * M * M])
        O = C0[k] @ bo.expm_eig(A)
        c2 = np.linalg.norm(C0[k], 2) ** 2
        worst[0] = max(worst[0], np.abs(D[k] - (O * occ[k]) @ O.conj().T).max()
                       / (2.0 * occ[k].max() * c2))
        Hmo = O.conj().T @ H[k] @ O
        L = occ[k][:, None] * Hmo - Hmo * occ[k][None, :]
        ref = bo.vars_of_grad(bo.grad_eq39(A, L))
        scale = 2.0 * occ[k].max() * np.linalg.norm(Hmo, 2)  # of L and its errors
        worst[1] = max(worst[1], np.abs(g[k] - ref).max() / (4.0 * scale))
    print(f"M={M} nk={nk} {kind}: exp(A) {worst[0]:.1e} g {worst[1]:.1e} (allowed {eps:.1e})")
    assert worst[0] <= eps and worst[1] <= eps
    s.close()
