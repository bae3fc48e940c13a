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
        return [[float(x) if "." in x or "e" in x else int(x) for x in ln.split()] for ln in res.stdout.splitlines()]
    return run


def test_sine_and_cosine(fix64):
    """Within 2^-51 in either form of the remainder (the phase's FP32 part 2^-58 revolutions, the remainder's
    rounding 2^-54, a few float-float roundings of that size), the exact negative half a revolution on, at
    random phases and around table boundaries."""
    mp = pytest.importorskip("mpmath")
    mp.mp.prec = 120
    rng = np.random.default_rng(1)
    ps = [int(x) for x in rng.integers(0, 2**63, 1500)]
    ps += [(k << 53) + (1 << 52) + d for k in range(0, 1024, 7) for d in (-1, 0, 1)]  # rounding of the index
    ps += [(k << 53) + d for k in (0, 1, 255, 256, 257, 511, 512, 513, 1023) for d in (-3, 0, 1, 2**31, 2**32 - 1)]
    ps = [p % 2**64 for p in ps]
    got = fix64([f"T {p:x}" for p in ps])
    opp = fix64([f"T {(p + 2**63) % 2**64:x}" for p in ps])
    bound = mp.mpf(2) ** -51
    for p, v, w in zip(ps, got, opp):
        a = 2 * mp.pi * mp.mpf(p) / 2**64
        for (h, f, i), exact in ((v[:3], mp.sin(a)), (v[3:], mp.cos(a))):
            assert abs((h + mp.mpf(f)) / 2**30 - exact) < bound, hex(p)
            assert abs((h + mp.mpf(i) / 2**24) / 2**30 - exact) < bound, hex(p)
            assert abs(f) < 1.8
        assert w == [-x for x in v], hex(p)


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
    """Products to 1.3 units (half of the rounding, and up to 0.7 of the left-out product of the low
    words); charges to half a unit of their 55 bits and exact within a factor of 4."""
    rng = np.random.default_rng(3)
    cases = [(int(h), int(l), int(b)) for h, l, b in zip(rng.integers(-2**30, 2**30, 500),
                                                         rng.integers(-20_000_000, 20_000_000, 500),
                                                         rng.integers(0, 2**60, 500))]
    cases += [(2**30, 21_000_000, 2**60 - 2**29 - 1), (-2**30, -21_000_000, 2**60 - 2**29 - 1), (5, 7, 0), (0, 0, 2**59)]
    for (h, l, b), (g,) in zip(cases, fix64([f"M {h} {l} {b}" for h, l, b in cases])):
        assert abs((h + Fraction(l, 2**24)) * Fraction(b, 2**30) - g) <= 1.3, (h, l, b)
    qs = [(float(q), e) for q in rng.uniform(0.0, 2.0, 200) for e in (0, 3, 40)] + [(1.0, 0), (0.0, 0), (5e-324, 0)]
    for (q, e), (g,) in zip(qs, fix64([f"Q {q!r} {e}" for q, e in qs])):
        d = abs(Fraction(q) * Fraction(2) ** (54 - e) - g)
        assert d <= Fraction(1, 2) and (d == 0 or q < 2.0 ** (e - 1)), (q, e)
