"""The FP64 real space at the edges of its tables, against the oracle's pair sum through rbe_npt_init and
rbe_water_init: cutoffs where erfc leaves the float range, tiny Lennard-Jones terms.  Tolerance 1e-11 of the
summed sizes of the energies' terms and of the largest force, as for the ordinary sizes: separations are exact to
2^-53 of the coordinates, up to 40 times the distance and 14 times amplified by u^-7."""
import numpy as np
import pytest

import oracle
import paper_2110_14362_gb300 as rbe
from gpu_util import cuda_device

pytestmark = pytest.mark.gpu


def _system(n, L, seed):
    """n^3 charges on a jittered grid."""
    rng = np.random.default_rng(seed)
    g = (np.arange(n) + 0.5) * (L / n)
    pos = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3) + rng.uniform(-0.15, 0.15, (n ** 3, 3)) * L / n
    q = rng.choice([-1.0, 1.0], n ** 3) * rng.uniform(0.3, 1.2, n ** 3)
    return np.mod(pos, L), q


def _params(rc, skin, sigma, eps):
    return rbe.NptParams(dt=0.001, kT=2.5, P_ext=0.0, gamma=1.0, gamma_V=1.0, M_V=1.0, rc=rc, qqr2e=1389.35, lj_sigma=sigma,
                         lj_eps=eps, max_disp=0.05, kspace=0, real=1, noise=0, barostat=0, skin=skin)


def _init(ctx, pos, q, L, prm):
    rep = rbe.NptReplica(pos, np.zeros_like(pos), q, np.full(len(q), 20.0), np.array([L, L, L]), prm, cuda_device())
    rep.init(ctx)
    ctx.sync()
    return rep.state()


@pytest.mark.parametrize("skin", [0.0, 0.7])
@pytest.mark.parametrize("alpha,rc,sigma,eps", [
    (0.2, 16.0, 2.0, 0.4),     # alpha rc^2 = 51
    (0.5, 12.0, 2.0, 0.4),     # 72
    (5.0, 10.0, 2.0, 0.4),     # 500
    (0.2, 7.0, 5e-4, 0.5),     # LJ far below the Coulomb terms
    (0.2, 7.0, 2.0, 1e-24),
])
def test_energies_beyond_the_tables(alpha, rc, sigma, eps, skin):
    L, box = 34.0, np.array([34.0, 34.0, 34.0])
    pos, q = _system(11, L, 3)
    with rbe.Context(box, alpha, 10, 1, rbe.RBE_FP64) as ctx:
        _, _, F, _, cell = _init(ctx, pos, q, L, _params(rc, skin, sigma, eps))
    F0, W0, Ec, El = oracle.pair_real(pos, q, box, alpha, rc, 1389.35, sigma, eps)
    assert np.abs(F - F0).max() <= 1e-11 * np.abs(F0).max()
    assert abs(cell[4] - np.trace(W0)) <= 1e-11 * max(abs(np.trace(W0)), np.abs(F0).max() * L)
    assert abs(cell[8] - Ec) <= 1e-11 * (abs(Ec) + 1389.35 * np.sum(q * q) / L)
    # each LJ term is at most eps (sigma / 2.1)^6 4 in size, the nearest pairs 2.1 apart at least; about 6 per particle
    assert abs(cell[9] - El) <= 1e-11 * (abs(El) + 4 * eps * (sigma / 2.1) ** 6 * 3 * len(q))


def test_water_energies_beyond_the_tables():
    n, L, alpha, rc = 6, 20.0, 0.7, 9.5  # alpha rc^2 = 63
    rng = np.random.default_rng(4)
    g = (np.arange(n) + 0.5) * (L / n)
    c = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3) + rng.uniform(-0.2, 0.2, (n ** 3, 3))
    half = np.radians(109.47) / 2
    mol = np.array([[0.0, 0.0, 0.0], [np.sin(half), 0.0, np.cos(half)], [-np.sin(half), 0.0, np.cos(half)]])
    pos = (c[:, None, :] + mol).reshape(-1, 3)
    q, m = np.tile([-0.8476, 0.4238, 0.4238], n ** 3), np.tile([15.9994, 1.008, 1.008], n ** 3)
    box = np.array([L, L, L])
    with rbe.Context(box, alpha, 10, 1, rbe.RBE_FP64) as ctx:
        rep = rbe.WaterReplica(pos, np.zeros_like(pos), q, m, box, _params(rc, 0.0, 3.166, 0.65), cuda_device())
        rep.init(ctx)
        ctx.sync()
        _, _, F, _, cell = rep.state()
    F0, _, *E = oracle.water_real(pos, q, box, alpha, rc, 1389.35, 3.166, 0.65)
    assert np.abs(F - F0).max() <= 1e-11 * np.abs(F0).max()
    for got, ref in ((cell[8], E[0]), (cell[9], E[1]), (cell[rbe.CELL_EXCL], E[2])):
        assert abs(got - ref) <= 1e-11 * (abs(ref) + 1389.35 * np.sum(q * q) / L), (got, ref)


@pytest.mark.parametrize("skin", [0.0, 0.7])
@pytest.mark.parametrize("gap", [1e-2, 1e-4, 1e-6])
def test_close_pairs(gap, skin):
    """Forces of charges `gap` apart to 1e-13 of their size: the difference of two FP64 coordinates is exact there, and
    the pair terms are a few roundings of it (the other pairs' forces are below 1e-5 of theirs)."""
    L, rc, box = 40.0, 7.0, np.array([40.0, 40.0, 40.0])
    rng = np.random.default_rng(6)
    a = (np.stack(np.meshgrid(*[[5.0, 18.0, 31.0]] * 3, indexing="ij"), -1).reshape(-1, 3) + rng.uniform(-1, 1, (27, 3)))
    v = rng.normal(size=a.shape)
    b = a + gap * v / np.linalg.norm(v, axis=1)[:, None]
    pos = np.stack([a, b], 1).reshape(-1, 3)
    q = rng.choice([-1.0, 1.0], len(pos)) * rng.uniform(0.3, 1.2, len(pos))
    with rbe.Context(box, 0.2, 10, 1, rbe.RBE_FP64) as ctx:
        _, _, F, _, cell = _init(ctx, pos, q, L, _params(rc, skin, 2.0, 0.0))
    F0, W0, Ec, _ = oracle.pair_real(pos, q, box, 0.2, rc, 1389.35, 2.0, 0.0)
    assert np.max(np.linalg.norm(F - F0, axis=1) / np.linalg.norm(F0, axis=1)) <= 1e-13
    assert abs(cell[4] - np.trace(W0)) <= 1e-13 * 1389.35 * len(a) * 1.44 / gap
    assert abs(cell[8] - Ec) <= 1e-13 * 1389.35 * len(a) * 1.44 / gap


def _replica(pos, q, L, eps, rc=5.0):
    return rbe.NptReplica(pos, np.zeros_like(pos), q, np.full(len(q), 20.0), np.array([L, L, L]), _params(rc, 0.0, 2.0, eps),
                          cuda_device())


def test_results_do_not_depend_on_earlier_parameters():
    """Twelve sets of Lennard-Jones parameters one after the other on one context, and the first and the last again: the
    bits of a context of its own for each."""
    L = 14.0
    pos, q = _system(6, L, 5)
    box = np.array([L, L, L])

    def run(ctx, k):
        rep = _replica(pos, q, L, 0.1 + 0.05 * k)
        rep.init(ctx)
        rep.step(ctx, 2)
        ctx.sync()
        return rep.state()

    with rbe.Context(box, 0.2, 10, 1, rbe.RBE_FP64) as shared:
        for k in [*range(12), 0, 11, 3]:
            with rbe.Context(box, 0.2, 10, 1, rbe.RBE_FP64) as own:
                for a, b in zip(run(shared, k), run(own, k)):
                    assert np.array_equal(a, b), k


def test_captured_steps_keep_their_tables():
    """A step captured with parameters that its context meets first in the capture, replayed after twenty other sets
    have been through the context: the bits of the same step launched directly."""
    import torch
    L = 14.0
    pos, q = _system(6, L, 5)
    box = np.array([L, L, L])
    with rbe.Context(box, 0.2, 10, 1, rbe.RBE_FP64) as ctx:
        rep = _replica(pos, q, L, 0.1)
        rep.init(ctx)
        rep.sys.params.lj_eps = 0.33
        rep.step(ctx, 3)
        ctx.sync()
        want = rep.state()
    stream = torch.cuda.Stream()
    with rbe.Context(box, 0.2, 10, 1, rbe.RBE_FP64) as ctx:
        ctx.set_stream(stream.cuda_stream)
        rep = _replica(pos, q, L, 0.1)
        torch.cuda.synchronize()
        rep.init(ctx)
        rep.sys.params.lj_eps = 0.33
        ctx.sync()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
            rep.step(ctx, 1)
        for k in range(20):
            other = _replica(pos, q, L, 0.5 + 0.01 * k)
            torch.cuda.synchronize()
            other.init(ctx)
            ctx.sync()
        with torch.cuda.stream(stream):
            for _ in range(3):
                g.replay()
        ctx.sync()
        for a, b in zip(want, rep.state()):
            assert np.array_equal(a, b)


def test_water_in_a_box_of_a_few_bonds():
    """Two molecules in a box of 3.6 bonds, hydrogens of both a bond outside it on opposite sides: the separation of their
    storage is 1.55 edges, and their nearest images are within rc."""
    L, rc, alpha = 3.6, 1.79, 1.0
    pos = np.array([[3.55, 0.5, 0.6], [4.55, 0.5, 0.6], [3.3, 1.4, 0.9], [0.03, 1.0, 0.8], [-0.97, 1.0, 0.8], [0.4, 1.9, 1.1]])
    q, m = np.tile([-0.8476, 0.4238, 0.4238], 2), np.tile([15.9994, 1.008, 1.008], 2)
    box = np.array([L, L, L])
    with rbe.Context(box, alpha, 10, 1, rbe.RBE_FP64) as ctx:
        rep = rbe.WaterReplica(pos, np.zeros_like(pos), q, m, box, _params(rc, 0.0, 1.2, 0.65), cuda_device())
        rep.init(ctx)
        ctx.sync()
        _, _, F, _, cell = rep.state()
    F0, _, *E = oracle.water_real(pos, q, box, alpha, rc, 1389.35, 1.2, 0.65)
    assert np.abs(F - F0).max() <= 1e-11 * np.abs(F0).max()
    for got, ref in ((cell[8], E[0]), (cell[9], E[1]), (cell[rbe.CELL_EXCL], E[2])):
        assert abs(got - ref) <= 1e-11 * (abs(ref) + 1389.35 * np.sum(q * q) / L), (got, ref)
