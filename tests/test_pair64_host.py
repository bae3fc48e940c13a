"""The tabulated pair terms of the FP64 real space (rbe_pair64.cuh), compiled for the host and checked
against multiple-precision arithmetic."""
import os
import shutil
import subprocess

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")
HERE = os.path.dirname(os.path.abspath(__file__))
EXE = os.path.join(HERE, "host", "_build", "pair64_main")


@pytest.fixture(scope="module")
def pair64():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    os.makedirs(os.path.dirname(EXE), exist_ok=True)
    src = os.path.join(HERE, "host", "pair64_main.cu")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-ffp-contract=off", "-o", EXE, src], check=True)

    def run(alpha, rc, sigma, eps, us):
        line = " ".join(repr(float(x)) for x in (alpha, rc, sigma, eps, *us)) + "\n"
        return subprocess.run([EXE], input=line, capture_output=True, text=True, check=True).stdout.splitlines()
    return run


@pytest.mark.parametrize("alpha,rc,sigma,eps", [(0.2, 7.0, 2.0, 0.5), (0.08, 10.0, 3.166, 0.65), (1.0, 4.0, 1.0, 1.0),
                                                (0.25, 8.0, 2.5, 0.3)])
def test_pair_terms(pair64, alpha, rc, sigma, eps):
    """Force factors to 2^-48 of their terms' sizes (eight roundings of FP64 and the first term left out,
    2^-58 times binomials up to 2^8), energies to 2^-43 (float-float with FP32 small terms), at random
    distances, at segment boundaries and next to the cutoff; below the table there is no segment.  The
    Coulomb terms' size is that of 1/r (erfc makes them smaller far out)."""
    mp.mp.prec = 120
    rng = np.random.default_rng(7)
    us = list(rng.uniform(0.4 * sigma, rc, 300) ** 2)
    e = 2.0 ** np.floor(np.log2(rc * rc))
    for b in (e, e / 2, e / 4, e / 8):
        for k in (0, 1, 63, 64, 127):
            x = b * (1 + k / 128)
            us += [x, np.nextafter(x, 0), np.nextafter(x, 1e9), b * (1 + (k + 0.5) / 128)]
    us = [u for u in us if u < rc * rc] + [float(np.nextafter(rc * rc, 0))]
    out = pair64(alpha, rc, sigma, eps, us)
    assert len(out) == len(us)
    for u, line in zip(us, out):
        f, ec, g, el = (mp.mpf(x) for x in line.split())
        U, a = mp.mpf(float(u)), mp.mpf(alpha)
        r, s = mp.sqrt(U), mp.sqrt(mp.mpf(alpha))
        E = mp.erfc(s * r) / r
        G = (E + 2 * s / mp.sqrt(mp.pi) * mp.exp(-a * U)) / U
        y3 = (mp.mpf(sigma * sigma) / U) ** 3
        F, L = 24 * mp.mpf(eps) * (2 * y3 * y3 - y3) / U, 4 * mp.mpf(eps) * (y3 * y3 - y3)
        assert abs(f - G) < 2.0 ** -48 / (U * r) * mp.mpf(min(1.0, float(G * U * r) + 1e-3)), u
        assert abs(ec - E) < 2.0 ** -43 / r, u
        assert abs(g - F) < 2.0 ** -48 * 24 * eps * (2 * y3 * y3 + y3) / U, u
        assert abs(el - L) < 2.0 ** -43 * 4 * eps * (y3 * y3 + y3), u
    top = 2.0 ** (np.floor(np.log2(rc * rc)) + 1)
    assert pair64(alpha, rc, sigma, eps, [np.nextafter(top / 256, 0), 1e-12]) == ["out", "out"]
