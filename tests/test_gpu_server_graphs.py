"""Requests long enough for their chunks to be replayed from a captured graph: the same bits as launched directly and as
the NPT step called on its own, on servers with one slot (the k-space on a side stream inside the capture), several,
and more than sixteen (launches in order), from a cell search and a neighbour list."""
import time

import numpy as np
import pytest

import oracle
import paper_2110_14362_gb300 as rbe
from gpu_util import cuda_device

pytestmark = pytest.mark.gpu
ALPHA, P, CHUNK = 0.2, 100, 2
REQS = [(6, 1, 11, 11), (9, 2, 22, 14), (8, 3, 33, 13), (7, 4, 44, 10), (6, 5, 55, 9)]  # side, seeds, steps (the last: 4 chunks)


def _system(n, seed):
    N = n ** 3
    L = (N / 0.1) ** (1 / 3)
    rng = np.random.default_rng(seed)
    g = (np.arange(n) + 0.5) * (L / n)
    pos = np.mod(np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3) + rng.uniform(-0.3, 0.3, (N, 3)), L)
    m = np.full(N, 20.0)
    mom = rng.normal(size=(N, 3)) * np.sqrt(oracle.KB * 300 * 100 * m)[:, None]
    return pos, mom, np.where(np.arange(N) % 2 == 0, 1.0, -1.0), m, np.array([L, L, L])


def _params(box, skin):
    return rbe.NptParams(dt=0.001, kT=oracle.KB * 300.0, P_ext=oracle.BAR, gamma=10.0, gamma_V=2.0,
                         M_V=oracle.piston_mass(0.5, 4.5e-5 / oracle.BAR, float(np.prod(box))), rc=6.0, qqr2e=oracle.QQR2E,
                         lj_sigma=2.0, lj_eps=0.5, max_disp=0.05, kspace=1, real=1, noise=1, barostat=1, skin=skin)


def _serve(precision, slots, skin, use_graphs):
    srv = rbe.Server(ALPHA, P, precision, max_slots=slots, chunk_steps=CHUNK, mem_budget=8 << 30, use_graphs=use_graphs)
    try:
        ids = []
        for n, sseed, pseed, steps in REQS:
            pos, mom, q, m, box = _system(n, sseed)
            ids.append(srv.submit(pos, mom, q, m, box, _params(box, skin), pseed, steps))
        end = time.monotonic() + 300.0
        while srv.progress(wait=True)[2] < len(ids):
            assert time.monotonic() < end, "serving loop did not finish"
        return [srv.result(i) for i in ids], srv.graph_replays()
    finally:
        srv.close()


@pytest.mark.parametrize("skin", [0.0, 0.4])
@pytest.mark.parametrize("slots", [1, 4, 9, 17])
@pytest.mark.parametrize("precision", [rbe.RBE_FP64, rbe.RBE_FP32_PHASE])
def test_replayed_chunks(precision, slots, skin):
    dev = cuda_device()
    graphs, replays = _serve(precision, slots, skin, True)
    direct, none = _serve(precision, slots, skin, False)
    assert replays == sum(r[3] // CHUNK for r in REQS[:4]) and none == 0
    for (n, sseed, pseed, steps), a, b in zip(REQS, graphs, direct):
        pos, mom, q, m, box = _system(n, sseed)
        with rbe.Context(box, ALPHA, P, pseed, precision) as ctx:
            rep = rbe.NptReplica(pos, mom, q, m, box, _params(box, skin), dev, step=0)
            rep.init(ctx, batch=0)
            rep.step(ctx, steps)
            ctx.sync()
            r, p, _, _, cell = rep.state()
        for x, y, z in zip(a, b, (r, p, cell)):
            assert np.array_equal(x, y) and np.array_equal(x, z)
