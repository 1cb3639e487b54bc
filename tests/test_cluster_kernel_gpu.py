"""The cluster kernel (k_fused.cu) against the oracle.  The one-kernel evaluator
(k_tile.cu) serves most fused calls by itself: a tuning of the default shape
keeps the calls here on the cluster kernel.  Tolerances of tests/cases.py."""
import numpy as np
import pytest
import torch

import oracle
from cases import check_maps, chi2_bound, make_obs, ogeom
from paper_1510_01815_gb300 import synth
from paper_1510_01815_gb300.synth import Geometry
from test_parity_gpu import CASES, _params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_1510_01815_gb300 import build, gbk
    build.build()
    return gbk


@pytest.fixture
def pinned(G):
    """Pins a geometry to the cluster kernel in its default shape."""
    done = []

    def pin(g):
        done.append(g)
        G.gbk_set_tuning(g, **G.gbk_get_tuning(g))

    yield pin
    for g in done:
        G.gbk_set_tuning(g, None)


@pytest.mark.parametrize("case", sorted(CASES))
def test_pinned_cluster_kernel_vs_oracle(G, pinned, case):
    g, p, ps = _params(case)
    ref = oracle.evaluate_batch(ogeom(g), ps)
    obs = make_obs(g, p, seed=3)
    dobs = G.Obs.from_numpy(obs.v, obs.s, obs.w_v, obs.w_s, obs.mask)
    d = torch.from_numpy(ps)
    pinned(g)
    maps = G.eval_maps(g, d).cpu().numpy()
    check_maps(maps, ref, ps, case)
    c, r = G.chi2(g, d, dobs, flags=G.PATH_FUSED, want_resid=True)
    for i in range(len(ps)):
        ref_c = oracle.chi2_maps(ref[i], obs)
        assert abs(float(c[i]) - ref_c) <= chi2_bound(ref[i], maps[i], obs, ref_c), i
        s = float((r[i].double() ** 2).sum())
        assert abs(float(c[i]) - s) <= 1e-5 * s + 1e-12


def test_pinned_full_size_image(G, pinned):
    """192 x 192 x 48 over a cluster of CTAs per model."""
    g = synth.FP_GEOM
    ps = synth.draw_fp_params(np.random.default_rng(12), 3, g)
    pinned(g)
    assert G.gbk_get_tuning(g)["cluster_ctas"] > 1
    maps = G.eval_maps(g, torch.from_numpy(ps)).cpu().numpy()
    check_maps(maps, oracle.evaluate_batch(ogeom(g), ps), ps, "full size")


def test_pinned_survey_vs_oracle(G):
    """A survey on one persistent cluster launch and on launches by group."""
    rng = np.random.default_rng(14)
    gal = synth.draw_survey(rng, 10, nxy_range=(24, 48)) + [
        (Geometry(110, 100, 24, 30.0, 0.0, 4.0, 40.0), synth.params(55, 50, 40, 50, 0, 150, 5, 40, 1, 12))]
    geoms, ps = [g for g, _ in gal], np.array([p for _, p in gal])
    shape = G.gbk_survey_get_tuning(geoms)
    ref = [oracle.evaluate(ogeom(g), p) for g, p in gal]
    try:
        for t in (shape, {"persistent": 0}):
            G.gbk_survey_set_tuning(geoms, **t)
            maps, _, _ = G.survey_eval(geoms, ps)
            for i in range(len(geoms)):
                check_maps(maps[i].cpu().numpy()[None], ref[i][None], ps[i:i + 1], "galaxy %d" % i)
    finally:
        G.gbk_survey_set_tuning(geoms, None)


@pytest.mark.parametrize("width", [0.2, 0.26, 0.46, 1.16, 4.0])
@pytest.mark.parametrize("reach", [0.3, 1.0, 2.0])
def test_valid_spectra_stay_valid(G, width, reach):
    """No form of the line sums loses a spectrum: spaxels whose oracle flux is
    above twice the threshold (cases.THRESH) have one, those below half of it
    have none."""
    g = Geometry(21, 18, 24, 20.0, 3.0, 2.0, 30.0)
    ps = synth.draw_fp_params(np.random.default_rng(17), 6, g, 4.0)
    ps[:, synth.SIG0] = width * g.dv
    ps[:, synth.VMAX] = reach * 0.5 * g.nz * g.dv
    ref = oracle.evaluate_batch(ogeom(g), ps)
    got = G.eval_maps(g, torch.from_numpy(ps)).cpu().numpy()
    assert (got[:, 0][ref[:, 0] > 2e-20] > 0).all()
    assert (got[:, 0][ref[:, 0] < 0.5e-20] == 0).all()
