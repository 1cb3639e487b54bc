"""Surveys whose galaxies take every kind of launch at once: images whole in
one CTA of each size with every PSF radius (0 to 8), images too large for one
CTA and PSFs too wide for it (the persistent cluster launch).  Maps and chi2
against the oracle (tolerances of tests/cases.py), the same bits in any order
of the galaxies, when evaluated again, and in a survey of a galaxy alone."""
import numpy as np
import pytest
import torch

import oracle
from cases import check_maps, chi2_bound, make_obs, ogeom
from paper_1510_01815_gb300 import synth
from paper_1510_01815_gb300.synth import Geometry

pytestmark = pytest.mark.gpu

FWHM = [0.0, 0.5, 1.1, 1.7, 2.3, 2.9, 3.5, 4.1, 4.7]  # PSF radii 0 .. 8
SIZES = [(12, 9), (30, 33), (47, 45), (64, 58), (95, 96)]  # 160 to 768 threads


def _geoms(large):
    out = [Geometry(nx, ny, 20 + 3 * i, 30.0, 0.0, FWHM[(i + 2 * k) % 9], 40.0, lsf_mode=i % 2)
           for k, (nx, ny) in enumerate(SIZES) for i in range(9 if k < 3 else 3)]
    if large:
        out += [Geometry(150, 140, 24, 30.0, 0.0, 2.9, 40.0), Geometry(24, 20, 24, 30.0, 0.0, 9.0, 40.0),
                Geometry(131, 128, 16, 30.0, 0.0, 4.7, 0.0)]
    return out


@pytest.mark.parametrize("large", [False, True])
def test_mixed_survey(large):
    from paper_1510_01815_gb300 import build, gbk as G
    build.build()
    geoms = _geoms(large)
    rng = np.random.default_rng(6)
    ps = np.array([synth.params(rng.uniform(0.4, 0.6) * g.nx, rng.uniform(0.4, 0.6) * g.ny, rng.uniform(0, 360),
                                rng.uniform(25, 70), rng.uniform(-5, 5), rng.uniform(80, 200), rng.uniform(1.5, 5),
                                rng.uniform(25, 60), 1.0, 0.12 * max(g.nx, g.ny) + 1.0) for g in geoms])
    obs = [make_obs(g, p, seed=i) for i, (g, p) in enumerate(zip(geoms, ps))]
    dobs = [G.Obs.from_numpy(o.v, o.s, o.w_v, o.w_s, o.mask) for o in obs]
    maps, c2, res = G.survey_eval(geoms, ps, dobs, want_resid=True)
    c2 = c2.cpu().numpy()
    for i, g in enumerate(geoms):
        ref = oracle.evaluate(ogeom(g), ps[i])
        got = maps[i].cpu().numpy()
        check_maps(got[None], ref[None], ps[i:i + 1], "galaxy %d" % i)
        ref_c = oracle.chi2_maps(ref, obs[i])
        assert abs(c2[i] - ref_c) <= chi2_bound(ref, got, obs[i], ref_c), i
    order = rng.permutation(len(geoms))
    m2, c3, r2 = G.survey_eval([geoms[i] for i in order], ps[order], [dobs[i] for i in order], want_resid=True)
    np.testing.assert_array_equal(c3.cpu().numpy(), c2[order])
    for k, i in enumerate(order):
        assert torch.equal(m2[k], maps[i]) and torch.equal(r2[k], res[i])
    for i in (0, 20, 30):
        _, alone, _ = G.survey_eval([geoms[i]], ps[i:i + 1], [dobs[i]], want_maps=False)
        assert float(alone[0]) == c2[i]
