"""gbk_jacobian asked for J alone (its launch carries no sums and twice the
threads) writes the same bits as the call that also reduces J^T J, J^T v and
chi2: the arithmetic of a spaxel does not depend on the launch shape."""
import numpy as np
import pytest
import torch

from cases import make_obs, model_params
from paper_1510_01815_gb300 import synth
from paper_1510_01815_gb300.synth import Geometry

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("g", [
    synth.SINGLE_GEOM,
    Geometry(9, 7, 4, 10.0, 0.0, 2.0, 60.0),      # fewer spaxels than threads
    Geometry(33, 23, 15, 20.0, 0.0, 3.0, 30.0),   # odd sizes, odd channels
    Geometry(72, 72, 40, 20.0, 0.0, 4.0, 30.0),   # halo rows read in the neighbours' shared memory
])
def test_jacobian_alone_has_the_same_bits(g):
    from paper_1510_01815_gb300 import build, gbk
    build.build()
    truth = synth.params(0.48 * g.nx, 0.52 * g.ny, 120.0, 55.0, 3.0, 120.0, 3.0, 40.0, 1.0, 0.15 * g.nx)
    ps = torch.from_numpy(np.ascontiguousarray(model_params(g, truth, 5, seed=13))).cuda()
    obs = make_obs(g, truth, seed=3)
    d = gbk.Obs.from_numpy(obs.v, obs.s, obs.w_v, obs.w_s, obs.mask)
    both = gbk.jacobian(g, ps, d, free=tuple(range(10)))[0]
    alone = torch.full_like(both, -7.0)
    gbk.gbk_jacobian(g, ps, d, tuple(range(10)), jac=alone)
    assert torch.equal(both, alone)
