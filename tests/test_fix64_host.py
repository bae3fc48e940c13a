"""The 64-bit fixed-point arithmetic of the FP64 path (rbe_fix64.cuh), compiled for the host and checked
against exact rational and multiple-precision arithmetic."""
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
EXE = os.path.join(HERE, "host", "_build", "fix64_main")


@pytest.fixture(scope="module")
def fix64():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    os.makedirs(os.path.dirname(EXE), exist_ok=True)
    src = os.path.join(HERE, "host", "fix64_main.cu")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-ffp-contract=off", "-o", EXE, src], check=True)

    def run(lines):
        res = subprocess.run([EXE], input="\n".join(lines) + "\n", capture_output=True, text=True, check=True)
        return [[int(x) for x in ln.split()] for ln in res.stdout.splitlines()]
    return run


def test_sine_and_cosine(fix64):
    """Within 2^-51 (the low part's grid 2^-53 and a few float-float roundings below it), the exact
    negative half a revolution on, at random phases and around every table boundary."""
    mp = pytest.importorskip("mpmath")
    mp.mp.prec = 120
    rng = np.random.default_rng(1)
    ps = [int(x) for x in rng.integers(0, 2**63, 1500)]
    ps += [(k << 53) + (1 << 52) + d for k in range(0, 1024, 7) for d in (-1, 0, 1)]  # rounding of the index
    ps += [(k << 53) + d for k in (0, 1, 255, 256, 257, 511, 512, 513, 1023) for d in (-3, 0, 1, 2**31, 2**32 - 1)]
    ps = [p % 2**64 for p in ps]
    got = fix64([f"T {p:x}" for p in ps])
    opp = fix64([f"T {(p + 2**63) % 2**64:x}" for p in ps])
    for p, (s, c), (s2, c2) in zip(ps, got, opp):
        a = 2 * mp.pi * mp.mpf(p) / 2**64
        assert abs(mp.mpf(s) / 2**62 - mp.sin(a)) < mp.mpf(2) ** -51, hex(p)
        assert abs(mp.mpf(c) / 2**62 - mp.cos(a)) < mp.mpf(2) ** -51, hex(p)
        assert (s2, c2) == (-s, -c), hex(p)


def test_fractions(fix64):
    """r / l in revolutions to 3 units of 2^-64 (half a unit of 1 / l per box length, and the rounding) for
    positions inside and a few boxes outside."""
    rng = np.random.default_rng(2)
    cases = []
    for l in (10.0, 80.0, 342.0, 1.0, 0.1, 3.3, 64.0, float(np.nextafter(64.0, 0)), float(np.nextafter(64.0, 65))):
        cases += [(float(r), l) for r in np.concatenate([rng.uniform(-2 * l, 2 * l, 60), [0.0, l, -l, 0.5 * l, 1e-30, l / 3]])]
    got = fix64([f"F {r!r} {l!r}" for r, l in cases])
    for (r, l), (g,) in zip(cases, got):
        d = (Fraction(r) / Fraction(l) * 2**64 - g) % 2**64
        assert min(d, 2**64 - d) <= 3, (r, l)


def test_products(fix64):
    """a |b| to one unit plus the truncation of |b| to 59 bits, and exactly antisymmetric in a for a power
    of two."""
    rng = np.random.default_rng(3)
    cases = [(int(a) - 2**61, float(b), -1) for a, b in zip(rng.integers(0, 2**62, 500), rng.uniform(0.0, 1.0, 500))]
    cases += [(2**62 - 1, 0.8476, -1), (-2**62 + 1, 1.0, 0), (2**62 - 1, 1e-3, -1), (12345, 0.0, 0), (-5, 5e-324, 0)]
    got = fix64([f"M {a} {b!r} {e}" for a, b, e in cases])
    for (a, b, e), (g,) in zip(cases, got):
        assert abs(Fraction(a, 2**62) * Fraction(b) / Fraction(2) ** (e + 1) * 2**57 - g) <= 1.25, (a, b, e)
    odd = [int(a) | 1 for a in rng.integers(0, 2**62, 300)]
    pos = fix64([f"M {a} 1.0 0" for a in odd])
    neg = fix64([f"M {-a} 1.0 0" for a in odd])
    assert all(x == -y for (x,), (y,) in zip(pos, neg))
