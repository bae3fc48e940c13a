"""The FP64 path's pair passes at the edges of their plan, against the oracle: frequency tiles of the rho
pass (512) and of the force pass (256), every number of frequency slices, charges over a wide range,
positions some boxes away.  Tolerance 2e-12 of the force RMS: the oracle's own phases m.s, up to 100
revolutions, are rounded at 2^-53 of their size, 7e-14 radians per term, and the largest of N random
sums of such terms stays within 30 of them."""
import numpy as np
import pytest

import oracle
import paper_2110_14362_gb300 as rbe
from gpu_util import cuda_device, rel_frob, rel_max_force

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,P", [(40, 513), (333, 512), (36000, 256), (70000, 257), (155000, 200)])
def test_fp64_plan_edges(N, P):
    import torch
    dev = cuda_device()
    rng = np.random.default_rng(N + P)
    box, alpha = np.array([21.0, 18.0, 25.5]), 0.4
    pos = rng.uniform(-1.5, 2.5, (N, 3)) * box
    q = rng.choice([-1.0, 1.0], N) * 10.0 ** rng.uniform(-5, 1, N)
    q[rng.integers(0, N, 3)] = 0.0
    F = torch.empty((N, 3), dtype=torch.float64, device=dev)
    W = torch.empty(9, dtype=torch.float64, device=dev)
    E = torch.empty(2, dtype=torch.float64, device=dev)
    with rbe.Context(box, alpha, P, 77, rbe.RBE_FP64) as ctx:
        ctx.forces_virial(torch.as_tensor(pos).to(dev), torch.as_tensor(q).to(dev), 5, F, W, E)
        ctx.sync()
        rho = ctx.rho()
    F0, W0, Ek0, Es0, m0, S0 = oracle.rbe_snapshot(pos, q, box, alpha, P, 77, 5)
    _, _, _, _, rho0 = oracle.rbe_kspace(pos, q, box, alpha, m0, S0 / P)
    assert np.max(np.abs(rho - rho0)) <= 2e-12 * np.sqrt(np.sum(q * q))
    assert rel_max_force(F.cpu().numpy(), F0) <= 2e-12 * max(1.0, np.max(np.abs(q)) / np.sqrt(np.mean(q * q)))
    assert rel_frob(W.cpu().numpy().reshape(3, 3), W0) <= 2e-12
    assert abs(E[0].item() - Ek0) <= 2e-12 * abs(Ek0)


def test_precision_switched_on_the_same_box():
    """FP32-phase first, FP64 next on the same box and context, and back: the bits of contexts of their own."""
    import torch
    dev = cuda_device()
    rng = np.random.default_rng(8)
    box, alpha, P, N = np.array([21.0, 18.0, 25.5]), 0.4, 100, 3000
    pos = torch.as_tensor(rng.uniform(0, 1, (N, 3)) * box).to(dev)
    q = torch.as_tensor(rng.choice([-1.0, 1.0], N)).to(dev)

    def evaluate(ctx):
        F = torch.empty((N, 3), dtype=torch.float64, device=dev)
        ctx.forces_virial(pos, q, 5, F)
        ctx.sync()
        return F.cpu().numpy()

    alone = {}
    for precision in (rbe.RBE_FP32_PHASE, rbe.RBE_FP64):
        with rbe.Context(box, alpha, P, 77, precision) as ctx:
            alone[precision] = evaluate(ctx)
    with rbe.Context(box, alpha, P, 77, rbe.RBE_FP32_PHASE) as ctx:
        for precision in (rbe.RBE_FP32_PHASE, rbe.RBE_FP64, rbe.RBE_FP32_PHASE, rbe.RBE_FP64):
            ctx.set_precision(precision)
            assert np.array_equal(evaluate(ctx), alone[precision])
