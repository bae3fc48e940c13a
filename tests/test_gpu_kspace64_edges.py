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
