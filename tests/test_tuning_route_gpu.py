"""The autotuners know the one-kernel evaluator: where it is the fastest the
geometry or survey keeps no tuning and its calls give the untuned bits (the
batches here are ones it serves in half the time of any cluster shape); a
tuning that the caller sets moves them to the cluster kernel."""
import numpy as np
import pytest
import torch

from paper_1510_01815_gb300 import synth
from paper_1510_01815_gb300.synth import Geometry

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_1510_01815_gb300 import build, gbk
    build.build()
    return gbk


def _obs(G, g):
    wv, ws = synth.weights((g.ny, g.nx), 5.0)
    z = np.zeros((g.ny, g.nx), np.float32)
    return G.Obs.from_numpy(z, z + 40.0, wv, ws, np.ones((g.ny, g.nx), np.uint8))


def test_autotuned_calls_keep_the_one_kernel_evaluator(G):
    g, n = synth.SINGLE_GEOM, 2048
    p = torch.from_numpy(synth.draw_fp_params(np.random.default_rng(1), n, g, 4.0)).cuda()
    obs = _obs(G, g)
    untuned, default = G.eval_maps(g, p), G.gbk_get_tuning(g)
    chi2 = G.chi2(g, p, obs, flags=G.PATH_FUSED)
    try:
        G.gbk_set_tuning(g, 4, 384, 1)
        assert not torch.equal(G.eval_maps(g, p), untuned)  # the kernels differ in their last bits
        best = G.gbk_autotune(g, p, obs, torch.empty(n, dtype=torch.float64, device="cuda"))
        assert {k: best[k] for k in default} == default == G.gbk_get_tuning(g)
        assert torch.equal(G.eval_maps(g, p), untuned)
        assert torch.equal(G.chi2(g, p, obs, flags=G.PATH_FUSED), chi2)
    finally:
        G.gbk_set_tuning(g, None)


def test_autotuned_chi2_of_large_images_leaves_the_maps_alone(G):
    """chi2 of an image too large for one CTA is the cluster kernel's without a
    workspace; its tuning does not move calls for the maps there."""
    g, n = Geometry(150, 140, 32, 20.0, 0.0, 3.0, 30.0), 64
    p = torch.from_numpy(synth.draw_fp_params(np.random.default_rng(2), n, g, 15.0)).cuda()
    untuned = G.eval_maps(g, p)
    try:
        best = G.gbk_autotune(g, p, _obs(G, g), torch.empty(n, dtype=torch.float64, device="cuda"))
        assert {k: best[k] for k in ("cluster_ctas", "threads", "persistent")} == G.gbk_get_tuning(g)
        assert torch.equal(G.eval_maps(g, p), untuned)
    finally:
        G.gbk_set_tuning(g, None)


def test_autotuned_survey_keeps_the_one_kernel_evaluator(G):
    gal = synth.draw_survey(np.random.default_rng(3), 512)
    geoms, ps = [g for g, _ in gal], np.array([p for _, p in gal])
    obs = [_obs(G, g) for g in geoms]
    untuned, chi2, _ = G.survey_eval(geoms, ps, obs)
    default = G.gbk_survey_get_tuning(geoms)
    try:
        G.gbk_survey_set_tuning(geoms, 0)
        maps, _, _ = G.survey_eval(geoms, ps, obs)
        assert not all(torch.equal(a, b) for a, b in zip(maps, untuned))
        dobs, _keep = G.obs_array(obs)
        scratch = torch.empty(len(geoms), dtype=torch.float64, device="cuda")
        ws = torch.empty(G.gbk_survey_workspace_bytes(geoms), dtype=torch.uint8, device="cuda")
        best = G.gbk_survey_autotune(geoms, torch.from_numpy(ps).cuda(), dobs, scratch, ws)
        assert {k: best[k] for k in default} == default == G.gbk_survey_get_tuning(geoms)
        maps, c, _ = G.survey_eval(geoms, ps, obs)
        assert all(torch.equal(a, b) for a, b in zip(maps, untuned)) and torch.equal(c, chi2)
    finally:
        G.gbk_survey_set_tuning(geoms, None)
