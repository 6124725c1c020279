"""The roots of the Householder scalars (csrc/roots.h) on the CPU against exact
ones, from single-precision seeds that are up to 2 units in the last place off:
no less accurate than sqrt(x) and 1 / sqrt(x) in FP64."""
import math
import os
import random
import shutil
import subprocess
from decimal import Decimal, getcontext

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_roots_against_exact_ones(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "roots_driver")
    # (no contraction: the products and sums are rounded as they are written)
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_2101_12597_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "roots_driver.cpp"), "-o", exe], check=True)
    rng = random.Random(5)
    xs, text = [], []
    for _ in range(20000):
        x = rng.uniform(1.0, 4.0) * 4.0 ** rng.randint(-49, 48)
        seed = np.float32(1.0 / math.sqrt(float(np.float32(x))))
        for _ in range(rng.randint(0, 2)):
            seed = np.nextafter(seed, np.float32(rng.choice([0.0, np.inf])))
        xs.append(x)
        text.append(f"{x.hex()} {float(seed).hex()}")
    out = subprocess.run([exe], input="\n".join(text), capture_output=True, text=True, check=True)
    getcontext().prec = 60
    worst = [0.0, 0.0, 0.0]
    for x, line in zip(xs, out.stdout.split("\n")):
        r, s = (float.fromhex(v) for v in line.split())
        root = Decimal(x).sqrt()
        for i, (v, exact) in enumerate([(r, 1 / root), (s, root), (1.0 / math.sqrt(x), 1 / root)]):
            worst[i] = max(worst[i], abs(float((Decimal(v) - exact) / Decimal(math.ulp(v)))))
    print("units in the last place: rsqrt %.3f, sqrt %.4f; 1 / sqrt(x) %.3f" % tuple(worst))
    assert worst[0] <= 1.0 and worst[1] <= 0.501 and worst[0] <= worst[2]
