"""The fixed-point separations of the FP64 real space (rbe_pair64.cuh), compiled for the host, against exact
rational arithmetic."""
import os
import shutil
import subprocess
from fractions import Fraction as Fr

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.parametrize("rc", [1.0, 6.999, 7.0, 10.0, np.nextafter(8.0, 0), 1e-3, 3e4])
@pytest.mark.parametrize("ratio", [2.0, 8.3, 4000.0])
def test_separations(tmp_path, rc, ratio):
    """Coordinates in [0, L] (and a little outside) and a neighbour within 1.06 rc of the first particle's image:
    the separations are exact to half a unit per coordinate below rc / 512 (exact otherwise), r^2 to below 2 units
    of the dropped parts plus 2^-1 per such rounding."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "pairfix_main")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-o", exe, os.path.join(HERE, "host", "pairfix_main.cu")], check=True)
    rng = np.random.default_rng(3)
    L = rc * ratio
    a = np.concatenate([rng.uniform(-0.1 * rc, L + 0.1 * rc, (200, 3)), rng.uniform(0, 1e-4 * rc, (20, 3)),
                        np.zeros((1, 3)), np.full((1, 3), L)])
    d = rng.normal(size=a.shape)
    d *= (rc * rng.uniform(0.01, 1.06, len(a)) / np.linalg.norm(d, axis=1))[:, None]
    b = a + d
    b[:, 0] += L
    text = "".join(" ".join(float(x).hex() for x in (rc, L, *p, *q)) + "\n" for p, q in zip(a, b))
    out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.splitlines()
    assert len(out) == len(a)
    for p, q, line in zip(a, b, out):
        s, *v = (int(x) for x in line.split())
        unit = Fr(2) ** s
        e = [(Fr(float(y)) - Fr(float(x)) - (Fr(float(L)) if t == 0 else 0)) * unit for t, (x, y) in enumerate(zip(p, q))]
        loose = [sum(abs(c) < rc / 512 and c != 0 for c in (x, y)) for x, y in zip(p, q)]
        for t in range(3):
            assert abs(v[t] - e[t]) <= Fr(1, 2) * loose[t]
        r2 = sum(x * x for x in e) / 2 ** 64
        assert -Fr(1, 2) * sum(loose) <= r2 - v[3] < 2 + Fr(1, 2) * sum(loose)
        assert 2 ** 58 <= v[4] < 2 ** 60
        assert abs(v[4] - (Fr(float(rc)) * unit) ** 2 / 2 ** 64) <= 129  # rc^2 rounded to FP64
