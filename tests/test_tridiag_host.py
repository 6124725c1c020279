"""The Sturm counts and sections of csrc/tridiag.h (the eigenvalues of iA(k)'s
tridiagonal form) against exact rational Sturm counts, on the CPU: matrices
whose entries determine every eigenvalue to its relative accuracy (zero
diagonals), graded over up to 60 orders of magnitude, and with off-diagonals
whose squares leave the range of FP64; for every number of section points."""
import os
import shutil
import subprocess
from fractions import Fraction as F

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2101_12597_gb300", "csrc")
EPS = F(1, 2 ** 53)


def exact_count(d, e, x):
    """Eigenvalues below x, in rational arithmetic (x no eigenvalue of a leading block)."""
    c, q = 0, None
    for j in range(len(d)):
        q = F(d[j]) - x - (F(e[j - 1]) ** 2 / q if j else 0)
        if q == 0:
            q = F(1, 2 ** 2000)
        c += q < 0
    return c


@pytest.fixture(scope="module")
def eigenvalues(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path_factory.mktemp("tri") / "tridiag_driver")
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", CSRC,
                    os.path.join(ROOT, "tests", "tridiag_driver.cpp"), "-o", exe], check=True)

    def run(d, e, P):
        text = f"{len(d)} {P}\n" + " ".join(f"{x!r}" for x in [*d, *e]) + "\n"
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True)
        return [float(x) for x in out.stdout.split()]
    return run


def cases():
    rng = np.random.default_rng(3)
    yield "random", [float(x) for x in rng.uniform(-0.3, 0.3, 14)], [float(x) for x in rng.uniform(0.01, 0.3, 13)]
    yield "zero diagonal", [0.0] * 14, [float(x) for x in rng.uniform(0.01, 0.4, 13)]
    yield "graded", [0.0] * 14, [0.4 * 10.0 ** (-4.0 * j) for j in range(13)]
    yield "small in between", [0.0] * 14, [0.3, 1e-25] * 6 + [0.2]
    # x lies far below the norm for rows on end: eight rows shrink a minor by 2^-1600
    yield "far below", [0.0] * 24, [0.4] + [2.0 ** -190, 2.0 ** -188] * 11
    yield "squares out of range", [0.25, -0.125] * 7, [0.25, 1e-170] * 6 + [0.125]


CASES = {name: (d, e) for name, d, e in cases()}


@pytest.mark.parametrize("P", [4, 8, 16, 32])
@pytest.mark.parametrize("which", list(CASES))
def test_eigenvalues_to_their_own_accuracy(which, P, eigenvalues):
    """A Sturm count is exact for a matrix whose e^2 differ by a few roundings
    each and whose d differ by roundings of d - x: with d = 0 every eigenvalue is
    known to some 4 n roundings of itself, else of the norm (below 1).  The
    sections' end adds 4."""
    d, e = CASES[which]
    n = len(d)
    lam = eigenvalues(d, e, P)
    assert lam == sorted(lam)
    zero = not any(d)
    for i, x in enumerate(lam):
        tol = (4 * n + 4) * EPS * (abs(F(x)) if zero else 1) + F(1, 2 ** 190)
        assert exact_count(d, e, F(x) - tol) <= i < exact_count(d, e, F(x) + tol), (i, x)
