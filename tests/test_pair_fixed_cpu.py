"""The fixed-point Hankel sequence of a disc pair (csrc/pair_fixed.cuh, compiled for the host)
against mpmath: J_s, Y_s times cos, sin of s phi for s = 0..2p, from the smallest distance it is
used at to the widest layouts, every direction, horizontal pairs included.

Tolerance, absolute on |h_s| < 1/4: a few units of 2^-53 from the FP64 distance and reciprocal
(1e-15), plus the phase's FP64 rounding z * 4 * 1.1e-16 times |h| = sqrt(2 / (pi z))."""
import math
import os
import random
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    out = str(tmp_path_factory.mktemp("pair") / "pair_fixed")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-I" + os.path.join(ROOT, "paper_1407_3868_gb300", "csrc"), "-o", out,
                    os.path.join(ROOT, "tests", "pair_fixed_host.cu")], check=True, capture_output=True)
    return out


@pytest.mark.parametrize("p", [0, 5, 11, 12, 15])
def test_sequence(program, p):
    mp = pytest.importorskip("mpmath")
    rng = random.Random(p)
    z0 = (26.0 if p <= 11 else 2.0 * p + 4.0) * (1 + 1e-6)
    pairs = []
    for i in range(24):
        k = rng.choice([1.0, 3.0, 3 * math.pi, 20.0])
        z = z0 * (1.0 if i == 0 else math.exp(rng.random() ** 2 * math.log(2.5e4 / z0)))
        a = [0.0, math.pi, math.pi / 2][i] if i < 3 else rng.uniform(-math.pi, math.pi)
        dx, dy = z / k * math.cos(a), z / k * math.sin(a)
        if i == 0:
            dx, dy = z / k, 0.0
        pairs.append((k, dx, dy))
    text = "\n".join(f"{k.hex()} {p} {dx.hex()} {dy.hex()}" for k, dx, dy in pairs)
    res = subprocess.run([program], input=text, capture_output=True, text=True, check=True)
    rows = iter(res.stdout.split("\n"))
    with mp.workdps(40):
        for k, dx, dy in pairs:
            z = mp.mpf(k) * mp.sqrt(mp.mpf(dx) ** 2 + mp.mpf(dy) ** 2)
            phi = mp.atan2(mp.mpf(dy), mp.mpf(dx))
            tol = 1e-15 + 4 * 1.1e-16 * float(z) * math.sqrt(2 / (math.pi * float(z)))
            for s in range(2 * p + 1):
                got = [mp.mpf(int(t)) / mp.mpf(2) ** 64 for t in next(rows).split()]
                h, c, sn = mp.hankel1(s, z), mp.cos(s * phi), mp.sin(s * phi)
                for g, e in zip(got, (h.real * c, h.real * sn, h.imag * c, h.imag * sn)):
                    assert abs(g - e) <= tol, (p, s, float(z))
