"""The FP64 path's phases (rbe_fix64.cuh) at frequencies of every size that a list or a batch can hold, compiled for
the host, against exact rational phases."""
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.parametrize("most", [1, 1000, 2**16, 2**16 + 1, 10**5, 3 * 10**5, 2**20, 10**7, 2**24 + 1, 2**31 - 1])
def test_phases_at_any_frequency(tmp_path, most):
    """Sine and cosine to 2^-51 (as at |m| = 1) and 2 pi |m| 2^-54: the low words' rounding 3 |m| 2^-58 revolutions,
    the three roundings of their FP32 sum 4.5 |m| 2^-57, those of m itself 1.5 |m| 2^-57.  The force pass's
    product adds 1.3 units (test_fix64_host)."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "phase_main")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-ffp-contract=off", "-o", exe,
                    os.path.join(HERE, "host", "phase_main.cu")], check=True)
    mp.mp.prec = 120
    rng = np.random.default_rng(most)
    l = np.array([21.0, 18.0, 25.5])
    m = rng.integers(-most, most, (400, 3), endpoint=True)
    m[:100] = rng.choice([-most, most], (100, 3))
    m[100:130, 1:] = 0
    if most == 2**31 - 1:
        m[0] = -2**31
    r = rng.uniform(-1, 2, (400, 3)) * l
    text = "".join(" ".join([*map(str, a), *(float(x).hex() for x in (*b, *l))]) + "\n" for a, b in zip(m.tolist(), r))
    out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.splitlines()
    assert len(out) == len(m)
    bound = mp.mpf(2) ** -51 + 2 * mp.pi * most * mp.mpf(2) ** -54
    for a, b, line in zip(m.tolist(), r, out):
        p = sum(k * Fraction(float(x)) / Fraction(float(y)) for k, x, y in zip(a, b, l)) % 1
        t = 2 * mp.pi * mp.mpf(p.numerator) / p.denominator
        sh, sl, ch, cl, prod = (mp.mpf(x) for x in line.split())
        assert abs((sh + sl) / 2**30 - mp.sin(t)) < bound, (a, b)
        assert abs((ch + cl) / 2**30 - mp.cos(t)) < bound, (a, b)
        b60 = 2**60 - 2**29 - 1
        assert abs(prod - mp.sin(t) * b60) < 1.3 + bound * b60, (a, b)
