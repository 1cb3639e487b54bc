"""Parameters at the ends of their accepted ranges: lengths whose squares or
ratios leave FP32's range in some unit must still give the oracle's maps
(tolerances of tests/cases.py)."""
import numpy as np
import pytest
import torch

import oracle
from cases import check_maps, ogeom
from paper_1510_01815_gb300 import synth
from paper_1510_01815_gb300.synth import params as P

pytestmark = pytest.mark.gpu

CASES = {
    # off the major axis (row 16) the deprojected radius is 6e6 px a row; the
    # minor axis (column 15) has the systemic velocity
    "edge_on_tiny_rt": P(15.0, 16.0, 90.0, 89.99999, 0.0, 200.0, 1e-12, 40.0, 1.0, 4.0),
    "edge_on_tinier_rt": P(15.0, 16.0, 90.0, 89.99999, 0.0, 200.0, 1e-30, 40.0, 1.0, 4.0),
    "far_centre_tiny_rt": P(-1e7, 16.0, 45.0, 80.0, 0.0, 200.0, 1e-12, 40.0, 1.0, 4e7),
    "rigid_rotation": P(15.3, 16.2, 30.0, 55.0, 0.0, 2e13, 1e12, 40.0, 1.0, 4.0),
}


@pytest.mark.parametrize("split", [False, True])
@pytest.mark.parametrize("case", sorted(CASES))
def test_extreme_parameters_vs_oracle(case, split):
    from paper_1510_01815_gb300 import build, gbk as G
    build.build()
    g, ps = synth.SINGLE_GEOM, CASES[case][None]
    ref = oracle.evaluate_batch(ogeom(g), ps)
    assert (ref[0, 0] > 1e-3).sum() >= 32  # the case has lines to compare
    maps = G.eval_maps(g, torch.from_numpy(ps), split=split).cpu().numpy()
    assert np.isfinite(maps).all()
    check_maps(maps, ref, ps, case)
