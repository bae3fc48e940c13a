"""The k-space of an NPT step beside its drift and real space, on the context's side stream: the same bits as
with kernel timing on, which keeps every launch in one stream's order."""
import numpy as np
import pytest

import oracle
import paper_2110_14362_gb300 as rbe
from paper_2110_14362_gb300 import inputs

from gpu_util import cuda_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [rbe.RBE_FP64, rbe.RBE_FP32_PHASE])
@pytest.mark.parametrize("N,skin,sampler", [(512, 0.0, rbe.RBE_SAMPLER_MH), (700, 0.8, rbe.RBE_SAMPLER_EXACT),
                                            (3000, 0.8, rbe.RBE_SAMPLER_OFFLINE)])
def test_side_stream_gives_the_same_bits(precision, N, skin, sampler):
    import torch
    pos, mom, q, m, box = inputs.npt_replica(N, 5)
    prm = rbe.NptParams(dt=0.001, kT=300.0 * oracle.KB, P_ext=oracle.BAR, gamma=10.0, gamma_V=2.0, M_V=oracle.piston_mass(0.5, 4.5e-5 / oracle.BAR, float(np.prod(box))), rc=0.45 * box.min(),
                        qqr2e=17.7, lj_sigma=2.0, lj_eps=0.5, max_disp=0.05, kspace=1, real=1, noise=1, barostat=1)
    prm.rc = min(prm.rc, 7.0)
    prm.skin = skin
    dev = cuda_device()
    out = []
    for in_order in (True, False, False):
        stream = torch.cuda.Stream(device=dev)
        with rbe.Context(box, 0.2, 100, 77, precision) as ctx:
            ctx.set_sampler(sampler)
            if in_order:
                ctx.set_kernel_timing(True)
            else:
                torch.cuda.synchronize()
                ctx.set_stream(stream.cuda_stream)
            rep = rbe.NptReplica(pos, mom, q, m, box, prm, dev)
            torch.cuda.synchronize()
            rep.init(ctx)
            rep.step(ctx, 4)
            ctx.sync()
            out.append(rep.state())
    for other in out[1:]:
        for a, b in zip(out[0], other):
            assert np.array_equal(a, b)
