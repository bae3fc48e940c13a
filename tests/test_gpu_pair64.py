"""The FP64 real space where its route changes: distances below the pair tables, charges outside their
range, a cutoff of half the box (image rounded per pair), a ninth set of parameters on one context (no
table left), cell search and list, against the oracle's pair sum.  Tolerance 1e-11 of the largest force and
of the summed term sizes: separations are exact to 2^-53 of the coordinates, up to 40 times the distance
and 14 times amplified by u^-7."""
import numpy as np
import pytest

import oracle
import paper_2110_14362_gb300 as rbe
from gpu_util import cuda_device

pytestmark = pytest.mark.gpu
ALPHA = 0.2


def _system(n, L, seed, close):
    """n^3 charges on a jittered grid; `close`: pairs moved to within 0.05 to 0.4 of each other."""
    rng = np.random.default_rng(seed)
    g = (np.arange(n) + 0.5) * (L / n)
    pos = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3) + rng.uniform(-0.15, 0.15, (n ** 3, 3)) * L / n
    for k in range(close):
        v = rng.normal(size=3)
        pos[2 * k + 1] = pos[2 * k] + v / np.linalg.norm(v) * rng.uniform(0.05, 0.4)
    q = rng.choice([-1.0, 1.0], n ** 3) * rng.uniform(0.3, 1.2, n ** 3)
    return np.mod(pos, L), q


def _check(ctx, pos, q, L, rc, skin, sigma, eps):
    box = np.array([L, L, L])
    prm = rbe.NptParams(dt=0.001, kT=2.5, P_ext=0.0, gamma=1.0, gamma_V=1.0, M_V=1.0, rc=rc, qqr2e=1389.35, lj_sigma=sigma,
                        lj_eps=eps, max_disp=0.05, kspace=0, real=1, noise=0, barostat=0, skin=skin)
    rep = rbe.NptReplica(pos, np.zeros_like(pos), q, np.full(len(q), 20.0), box, prm, cuda_device())
    rep.init(ctx)
    ctx.sync()
    _, _, F, _, cell = rep.state()
    F0, W0, Ec, El = oracle.pair_real(pos, q, box, ALPHA, rc, 1389.35, sigma, eps)
    assert np.abs(F - F0).max() <= 1e-11 * np.abs(F0).max()
    assert abs(cell[4] - np.trace(W0)) <= 1e-11 * max(abs(np.trace(W0)), np.abs(F0).max() * L)
    assert abs(cell[8] - Ec) <= 1e-11 * (abs(Ec) + 1389.35 * np.sum(q * q) / L)
    assert abs(cell[9] - El) <= 1e-11 * (abs(El) + eps * len(q))


@pytest.mark.parametrize("n,L,rc,skin,sigma,eps,close,scale", [
    (7, 15.0, 7.0, 0.0, 0.3, 0.5, 40, 1.0),     # below the table, cell search with 2 cells per axis
    (9, 24.0, 7.0, 1.0, 0.3, 0.5, 40, 1.0),     # below the table, list
    (6, 13.0, 6.5, 0.0, 2.0, 0.4, 0, 1.0),      # rc = l / 2
    (6, 13.0, 6.5, 0.0, 2.0, 0.0, 0, 1e-25),    # charges outside the table's range, no LJ
    (9, 22.0, 5.0, 0.7, 2.0, 0.4, 0, 1e25),
    (12, 30.0, 4.0, 0.0, 2.0, 0.4, 0, 1.0),     # 7 cells per axis
])
def test_pair_routes(n, L, rc, skin, sigma, eps, close, scale):
    pos, q = _system(n, L, 3, close)
    with rbe.Context([L, L, L], ALPHA, 10, 1, rbe.RBE_FP64) as ctx:
        _check(ctx, pos, q * scale, L, rc, skin, sigma, eps)


def test_many_parameter_sets():
    pos, q = _system(6, 14.0, 5, 0)
    with rbe.Context([14.0, 14.0, 14.0], ALPHA, 10, 1, rbe.RBE_FP64) as ctx:
        for k in list(range(10)) + [0, 9]:
            _check(ctx, pos, q, 14.0, 5.0 + 0.2 * k, 0.0, 2.0, 0.4)


@pytest.mark.parametrize("skin", [0.0, 0.6])
@pytest.mark.parametrize("N", [1, 2, 33, 609, 1217, 2433, 3801])
def test_last_rounds(N, skin):
    """Particle counts around the blocks' rounds (particles shared by 1, 2, 4, 8 or 16 warps, idle warps and
    blocks); cells out of reach at 3 to 8 cells per axis."""
    n = int(np.ceil(N ** (1 / 3)))
    L = max(12.0, n * 2.2)
    pos, q = _system(n, L, 11, 0)
    keep = np.random.default_rng(N).permutation(n ** 3)[:N]
    with rbe.Context([L, L, L], ALPHA, 10, 1, rbe.RBE_FP64) as ctx:
        if N > 1:
            _check(ctx, pos[keep], q[keep], L, 4.0, skin, 2.0, 0.4)
        else:
            rep_pos = pos[keep] * 0 + [0.0, L - 1e-12, 5.0]
            prm = rbe.NptParams(dt=0.001, kT=2.5, P_ext=0.0, gamma=1.0, gamma_V=1.0, M_V=1.0, rc=4.0, qqr2e=1389.35, lj_sigma=2.0,
                                lj_eps=0.4, max_disp=0.05, kspace=0, real=1, noise=0, barostat=0, skin=skin)
            rep = rbe.NptReplica(rep_pos, rep_pos * 0, q[keep], np.full(1, 20.0), np.array([L, L, L]), prm, cuda_device())
            rep.init(ctx)
            ctx.sync()
            assert np.all(rep.state()[2] == 0.0)
