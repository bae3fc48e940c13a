"""The range of the FP64 real space's tables (rbe_pair64.cuh), compiled for the host, against multiple-precision
arithmetic: large alpha rc^2, where erfc leaves the float range, and tiny Lennard-Jones terms."""
import os
import shutil
import subprocess

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def energies(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path_factory.mktemp("pair64") / "range_main")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-ffp-contract=off", "-o", exe,
                    os.path.join(HERE, "host", "pair64_range_main.cu")], check=True)

    def run(alpha, rc, sigma, eps, us):
        line = " ".join(repr(float(x)) for x in (alpha, rc, sigma, eps, *us)) + "\n"
        return subprocess.run([exe], input=line, capture_output=True, text=True, check=True).stdout.splitlines()
    return run


@pytest.mark.parametrize("ar2,rc,sigma,eps", [
    (16.0, 10.0, 3.0, 0.5), (20.0, 10.0, 3.0, 0.5), (50.0, 10.0, 3.0, 0.5), (52.0, 10.0, 3.0, 0.5), (60.0, 1.0, 0.3, 0.5),
    (100.0, 10.0, 3.0, 0.5), (200.0, 7.0, 2.0, 0.5), (1000.0, 1e4, 3e3, 0.5), (40.0, 1e4, 3e3, 0.5),
    (9.8, 7.0, 0.02, 0.5), (9.8, 7.0, 5e-4, 0.5), (9.8, 7.0, 2.0, 1e-24), (9.8, 7.0, 2.0, 1e-15), (9.8, 7.0, 1e-9, 1e9),
    (9.8, 7.0, 0.0, 0.5), (9.8, 7.0, 2.0, 0.0)])
def test_energies_over_the_range(energies, ar2, rc, sigma, eps):
    """Where the table is used: Coulomb energies to 2^-43 of 1/r and, of their own size, to 2^-40 and the series'
    first term left out, 2 (alpha h)^8 / 8! with alpha h = alpha u / 256 (erfc up to alpha u = 40); LJ energies to
    2^-43 of their terms' sizes.  Below alpha u = 39 and with ordinary LJ sizes the table is used."""
    mp.mp.prec = 120
    alpha = ar2 / rc ** 2
    rng = np.random.default_rng(5)
    us = list(rc * rc * rng.uniform(0.005, 1.0, 400)) + [rc * rc * (1 - 2.0 ** -k) for k in (1, 2, 3, 7, 8, 20, 50)]
    us += [x for k in range(60) if (x := 2 ** (1 / 3) * sigma * sigma * (1 + 1e-4 * (k - 30))) < rc * rc and x > rc * rc / 100]
    out = energies(alpha, rc, sigma, eps, us)
    assert len(out) == len(us)
    bottom = 2.0 ** (np.floor(np.log2(rc * rc)) + 1) / 256  # of the table
    ordinary = eps == 0.0 or (sigma >= 0.01 * rc / 7 and eps >= 0.1)
    for u, line in zip(us, out):
        if line == "direct":
            assert not (bottom <= u < 39.0 / alpha and ordinary), u
            continue
        ec, el = (mp.mpf(x) for x in line.split())
        U, a = mp.mpf(float(u)), mp.mpf(alpha)
        E = mp.erfc(mp.sqrt(a * U)) / mp.sqrt(U)
        assert abs(ec - E) < 2.0 ** -43 / mp.sqrt(U), u
        assert abs(ec - E) < (2.0 ** -40 + 2 * (alpha * u / 256) ** 8 / 40320) * E, u
        y3 = (mp.mpf(sigma * sigma) / U) ** 3
        assert abs(el - 4 * mp.mpf(eps) * (y3 * y3 - y3)) <= 2.0 ** -43 * 4 * eps * (y3 * y3 + y3), u


@pytest.fixture(scope="module")
def sums(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path_factory.mktemp("pair64") / "energy_main")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-ffp-contract=off", "-o", exe,
                    os.path.join(HERE, "host", "pair64_energy_main.cu")], check=True)
    return lambda text: subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.splitlines()


@pytest.mark.parametrize("alpha,rc,sigma,eps", [(0.2, 7.0, 2.0, 0.5), (0.08, 10.0, 3.166, 0.65), (1.0, 4.0, 1.0, 1.0)])
def test_energies_to_fp64(sums, alpha, rc, sigma, eps):
    """The energies as the pair kernels sum them, beside the float-float form's 2^-45 to 2^-47: Coulomb to 2^-51.5 of
    1/r (the constant term's rounding and erfc's, 1.5 2^-53; the rest, 2^-8 of it, to 2^-45), LJ to 2^-48.5 of its
    terms (the cubic term, 84 2^-24 of the constant one, in FP32)."""
    mp.mp.prec = 120
    us = np.random.default_rng(9).uniform(0.4 * sigma, rc, 1000) ** 2
    for u, line in zip(us, sums(" ".join(repr(float(x)) for x in (alpha, rc, sigma, eps, *us)) + "\n")):
        ec, dc, el, dl = (mp.mpf(x) for x in line.split())
        U = mp.mpf(float(u))
        r, y3 = mp.sqrt(U), (mp.mpf(sigma * sigma) / U) ** 3
        assert abs(ec + dc - mp.erfc(mp.sqrt(mp.mpf(alpha)) * r) / r) < 2.0 ** -51.5 / r, u
        assert abs(el + dl - 4 * mp.mpf(eps) * (y3 * y3 - y3)) < 2.0 ** -48.5 * 4 * eps * (y3 * y3 + y3), u


def test_square_sums_are_unbiased(sums):
    """Over random separations the rounded square sum is neither above nor below in the mean: 0.05 units, seven times
    the deviation of 4000 such roundings (0.45 each: the sum's 1/sqrt(12), the dropped squares' 0.13 and the halves)."""
    mp.mp.prec = 150
    d = np.random.default_rng(2).integers(-2**61, 2**61, (4000, 3))
    out = sums("".join("R %d %d %d\n" % tuple(x) for x in d.tolist()))
    err = [float(int(n) - mp.mpf(sum(c * c for c in x)) / 2**64) for n, x in zip(out, d.tolist())]
    assert abs(np.mean(err)) < 0.05
