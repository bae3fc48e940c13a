"""The constraint solves of the rigid-water drift: FP32 Newton steps (all but the last four iterations allowed)
and FP64 ones end at the same positions.  A stop at |r^2 - d^2| <= 1e-14 d^2 leaves 1e-14 A in a site, which is
m 1e-14 / (dt/2), below 1e-9 g/mol A/ps, in a momentum; a step in between amplifies it by less than ten."""
import numpy as np
import pytest

import paper_2110_14362_gb300 as rbe
from gpu_util import cuda_device
from test_gpu_water import ALPHA, P, SEED, _box_1gcc, _params, _waters

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_side", [1, 3, 5])  # 1, 27 and 125 molecules: blocks of 32 with and without a rest
@pytest.mark.parametrize("noise", [0, 1])
def test_fp32_and_fp64_solves_agree(n_side, noise):
    L = max(13.0, _box_1gcc(n_side ** 3))
    pos, mom, q, m, box = _waters(n_side, L, 3)
    prm, _ = _params(L, 6.0, noise=noise)
    dev = cuda_device()
    out = []
    for max_iter in (4, 6, 500):  # FP64 throughout; two FP32 solves first; FP32 throughout
        with rbe.Context(box, ALPHA, P, SEED, rbe.RBE_FP64) as ctx:
            rep = rbe.WaterReplica(pos, mom * 0.3, q, m, box, prm, dev, wp=rbe.water_params(shake_max_iter=max_iter))
            rep.init(ctx)
            rep.step(ctx, 2)
            ctx.sync()
            out.append(rep.state())
    for r, p, F, box_now, cell in out[1:]:
        d = r - out[0][0]
        assert np.abs(d - L * np.round(d / L)).max() < 1e-12
        assert np.abs(p - out[0][1]).max() < 1e-8
        mol = r.reshape(-1, 3, 3)
        assert np.abs(np.linalg.norm(mol[:, 1:] - mol[:, :1], axis=2) - 1.0).max() < 1e-13
