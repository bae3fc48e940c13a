"""The FP64 k-space at inputs outside the ordinary ones."""
import numpy as np
import pytest

import oracle
import paper_2110_14362_gb300 as rbe
from gpu_util import cuda_device, rel_max_force

pytestmark = pytest.mark.gpu
BOX = np.array([21.0, 18.0, 25.5])


def _weighted(pos, q, m, w, box=BOX, alpha=0.4):
    """(F, W, E, rho) of one weighted evaluation on an FP64 context; no check of its status."""
    import torch
    dev = cuda_device()
    N = len(q)
    F = torch.empty((N, 3), dtype=torch.float64, device=dev)
    W = torch.empty(9, dtype=torch.float64, device=dev)
    E = torch.empty(2, dtype=torch.float64, device=dev)
    with rbe.Context(box, alpha, 10, 1, rbe.RBE_FP64) as ctx:
        ctx.weighted(torch.as_tensor(pos).to(dev), torch.as_tensor(q).to(dev),
                     torch.as_tensor(np.ascontiguousarray(m, dtype=np.int32)).to(dev), torch.as_tensor(w).to(dev), F, W, E)
        torch.cuda.synchronize()
        status = rbe.RBE_OK
        try:
            ctx.sync()
        except rbe.RBEError as err:
            status = err.status
        rho = ctx.rho(len(w))
    return F.cpu().numpy(), W.cpu().numpy().reshape(3, 3), E.cpu().numpy(), rho, status


@pytest.mark.parametrize("N,K", [(50, 1), (400, 300), (5000, 60)])
def test_weights_of_both_signs(N, K):
    """Forces, energy and virial against the oracle; 2e-12 of the force RMS as in test_gpu_kspace64."""
    rng = np.random.default_rng(N)
    pos, q = rng.uniform(0, 1, (N, 3)) * BOX, rng.choice([-1.0, 1.0], N)
    m = rng.integers(-12, 13, (K, 3))
    m[~m.any(1)] = 1
    w = rng.normal(size=K)
    w[0] = -0.7
    F, W, E, rho, status = _weighted(pos, q, m, w)
    F0, W0, Ek0, _, rho0 = oracle.rbe_kspace(pos, q, BOX, 0.4, m, w)
    assert status == rbe.RBE_OK
    assert np.max(np.abs(rho - rho0)) <= 2e-12 * np.sqrt(N)
    assert rel_max_force(F, F0) <= 2e-12
    # energy and virial are sums of terms of both signs: 2e-12 of the sums of their sizes
    kk = np.sum((2 * np.pi * m / BOX) ** 2, axis=1)
    e = 2 * np.pi / np.prod(BOX) * np.abs(w) * np.abs(rho0) ** 2 / kk
    assert abs(E[0] - Ek0) <= 2e-12 * e.sum()
    assert np.linalg.norm(W - W0) <= 2e-12 * np.sum(e * (4 + kk / 0.8))


def _exact(S, q, m, w, box, alpha):
    """(F, E_k, rho, bound of the force) for positions S 2^-64 box (S uint64): the phases in wrapping integers."""
    p = sum(m[:, t].astype(np.int64).astype(np.uint64)[None, :] * S[:, t][:, None] for t in range(3))
    t = 2 * np.pi * (p.astype(np.int64) / 2.0 ** 64)
    c, s = np.cos(t), np.sin(t)
    rho = q @ c + 1j * (q @ s)
    k = 2 * np.pi * m / box
    kk = np.sum(k * k, axis=1)
    beta = w * 4 * np.pi / (np.prod(box) * kk)
    F = q[:, None] * ((s * (beta * rho.real) - c * (beta * rho.imag)) @ k)
    size = np.abs(q).max() * np.max(np.sum(np.abs(beta * np.abs(rho))[:, None] * np.abs(k), axis=0))
    return F, 2 * np.pi / np.prod(box) * np.sum(w * np.abs(rho) ** 2 / kk), rho, size


def _dyadic(N, box, seed):
    """Positions on a grid of 2^-50 box, exact in FP64 for boxes that are powers of two, and the same times 2^64 / box."""
    S = np.random.default_rng(seed).integers(0, 2 ** 50, (N, 3), dtype=np.int64)
    return S / 2.0 ** 50 * box, S.astype(np.uint64) << np.uint64(14)


@pytest.mark.parametrize("N,K,most", [(60, 300, 10**7), (60, 600, 3 * 10**5), (40000, 20, 2**20), (3000, 40, 2**31 - 1),
                                      (70000, 8, 10**6)])
def test_large_frequencies(N, K, most):
    """Lists with |m| up to any 32-bit size, small rows among them; each sine to 2 pi |m| 2^-54 (test_phase_host)
    in rho and again in the force, beside 2e-12 of the sums of the terms' sizes."""
    box = np.array([16.0, 32.0, 8.0])
    rng = np.random.default_rng(K)
    pos, S = _dyadic(N, box, N)
    q = rng.choice([-1.0, 1.0], N) * rng.uniform(0.5, 1.0, N)
    m = rng.integers(-most, most, (K, 3), endpoint=True)
    m[::3] = rng.integers(1, 12, (len(m[::3]), 3))
    w = rng.uniform(0.5, 1.0, K) * np.sum(m.astype(float) ** 2, axis=1) ** 0.5  # every size counts in the force
    F, _, E, rho, status = _weighted(pos, q, m, w, box)
    F0, E0, rho0, size = _exact(S, q, m, w, box, 0.4)
    err = 2 * np.pi * most * 2.0 ** -54 + 2e-12
    assert status == rbe.RBE_OK
    assert np.max(np.abs(rho - rho0)) <= err * np.sum(np.abs(q))
    # sin(theta_i - arg rho): the phase's error and that of arg rho, N err / |rho|
    assert np.max(np.abs(F - F0)) <= size * err * (1 + np.sum(np.abs(q)) / np.abs(rho0).min())
    assert abs(E[0] - E0) <= 2 * err * E0 * np.sum(np.abs(q)) / np.abs(rho0).min()


def test_large_frequencies_sampled():
    """A batch of a box where the sampler draws |m| of some 1e5."""
    import torch
    dev = cuda_device()
    box, alpha, P, N = np.array([2.0 ** 18, 2.0 ** 18, 2.0 ** 17]), 1.0, 64, 500
    pos, S = _dyadic(N, box, 2)
    q = np.random.default_rng(3).choice([-1.0, 1.0], N)
    F = torch.empty((N, 3), dtype=torch.float64, device=dev)
    with rbe.Context(box, alpha, P, 9, rbe.RBE_FP64) as ctx:
        ctx.forces_virial(torch.as_tensor(pos).to(dev), torch.as_tensor(q).to(dev), 4, F)
        ctx.sync()
        rho = ctx.rho()
        m, total = ctx.sample_k(4)
    m = np.asarray(m)
    assert np.abs(m).max() > 10**5
    F0, _, rho0, size = _exact(S, q, m, np.full(P, total / P), box, alpha)
    err = 2 * np.pi * np.abs(m).max() * 2.0 ** -54 + 2e-12
    assert np.max(np.abs(rho - rho0)) <= err * N
    assert np.max(np.abs(F.cpu().numpy() - F0)) <= size * err * (1 + N / np.abs(rho0).min())


@pytest.mark.parametrize("e", [-560, -505, 505, 560])
def test_rho_whose_square_leaves_fp64(e):
    """Forces are linear in rho and in the weights: charges times 2^e and weights times 2^(-2 e + 100) give forces
    times 2^100, whatever |rho|^2 does (it is 0 or infinite at 2^(+-1120), subnormal terms left out)."""
    rng = np.random.default_rng(1)
    N, K = 300, 40
    pos, q = rng.uniform(0, 1, (N, 3)) * BOX, rng.choice([-1.0, 1.0], N)
    m, w = rng.integers(1, 12, (K, 3)), rng.uniform(0.5, 1.0, K)
    F, _, _, _, _ = _weighted(pos, q, m, w)
    G, _, _, _, _ = _weighted(pos, np.ldexp(q, e), m, np.ldexp(w, max(-1000, min(1000, -2 * e + 100))))
    back = 100 if abs(2 * e - 100) <= 1000 else 2 * e + (1000 if e < 0 else -1000)
    assert rel_max_force(np.ldexp(G, -back), F) <= 1e-13


@pytest.mark.parametrize("N,K", [(700, 600), (40000, 20), (70000, 8)])
@pytest.mark.parametrize("what", ["position", "infinite position", "charge", "infinite charge", "far position", "zero row",
                                  "weight"])
def test_non_finite_inputs_show(what, N, K):
    """One input that is not finite (or whose r / l is not): no force, energy or virial is, and the status tells.  A
    frequency of zero or a weight of NaN leaves rho alone."""
    rng = np.random.default_rng(1)
    box = np.array([0.4, 0.5, 0.3])
    pos, q = rng.uniform(0, 1, (N, 3)) * box, np.where(np.arange(N) % 2, 1.0, -1.0)
    m, w = rng.integers(1, 12, (K, 3)), rng.uniform(0.5, 1.0, K)
    i, l = int(rng.integers(N)), int(rng.integers(K))
    if what.endswith("position"):
        pos[i, 1] = {"position": np.nan, "infinite position": np.inf, "far position": 1.2e308}[what]
    elif what.endswith("charge"):
        q[i] = np.nan if what == "charge" else np.inf
    elif what == "weight":
        w[l] = np.nan
    else:
        m[l] = 0
    F, W, E, rho, status = _weighted(pos, q, m, w, box=box, alpha=400.0)
    assert status == rbe.RBE_ENONFINITE
    assert not np.isfinite(F).any() and not np.isfinite(E[0]) and not np.isfinite(W).any()
    assert np.isfinite(rho).all() if what in ("zero row", "weight") else not np.isfinite(rho).any()


@pytest.mark.parametrize("N,K", [(60, 300), (3000, 40), (40000, 20), (70000, 8)])
def test_lists_equal_batches(N, K):
    """A sampled batch (its |m| bounded by the tables) and the same frequencies as a list (bounded by nothing): the same
    bits."""
    import torch
    dev = cuda_device()
    rng = np.random.default_rng(N)
    pos, q = rng.uniform(0, 1, (N, 3)) * BOX, rng.choice([-1.0, 1.0], N) * rng.uniform(0.5, 1.0, N)
    F = torch.empty((N, 3), dtype=torch.float64, device=dev)
    W = torch.empty(9, dtype=torch.float64, device=dev)
    E = torch.empty(2, dtype=torch.float64, device=dev)
    with rbe.Context(BOX, 0.4, K, 9, rbe.RBE_FP64) as ctx:
        ctx.forces_virial(torch.as_tensor(pos).to(dev), torch.as_tensor(q).to(dev), 4, F, W, E)
        ctx.sync()
        rho = ctx.rho()
        m, S = ctx.sample_k(4)
    F1, W1, E1, rho1, _ = _weighted(pos, q, np.asarray(m), np.full(K, S / K))
    assert np.array_equal(F.cpu().numpy(), F1) and np.array_equal(W.cpu().numpy().reshape(3, 3), W1)
    assert np.array_equal(E.cpu().numpy(), E1) and np.array_equal(rho, rho1)
