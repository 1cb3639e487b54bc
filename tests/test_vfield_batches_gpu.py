"""Velocity fields in batches that take a cluster of CTAs per model and in
batches that take a CTA per model: chi2, residuals, Jacobian and normal
equations of the same models are the same to the bit, and so are fits."""
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


def _params(nx, ny, n, rng):
    p = np.tile([0.45 * nx, 0.55 * ny, 30.0, 50.0, 5.0, 200.0, 4.0, 30.0, 1.2, 0.9], (n, 1))
    p[:, synth.PA] = rng.uniform(0, 360, n)
    p[:, synth.INCL] = rng.uniform(30, 70, n)
    return p


def _obs(G, nx, ny, rng, v=None):
    f = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    shape = (ny, nx)
    v = rng.normal(0, 80, shape) if v is None else v + rng.normal(0, 5, shape)
    return G.Obs(f(v), f(rng.uniform(20, 40, shape)), f(rng.uniform(0.1, 0.3, shape)), f(rng.uniform(0.1, 0.3, shape)),
                 torch.from_numpy((rng.uniform(size=shape) > 0.1).astype(np.uint8)).cuda())


@pytest.mark.parametrize("model", [1, 2])
@pytest.mark.parametrize("nx,ny", [(7, 5), (33, 31), (64, 64), (200, 171)])
def test_batches_agree(G, nx, ny, model):
    rng = np.random.default_rng(nx)
    g = Geometry(nx, ny, 1, 10.0, model=model)
    n = 320
    p = _params(nx, ny, n, rng)
    p[2, synth.RT] = -1.0  # outside the parameter domain: NaN
    obs = _obs(G, nx, ny, rng)
    cot = torch.randn((n, 2, ny, nx), device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    free, got = tuple(range(10)), []
    for m in (3, 17, n):
        d = torch.from_numpy(p[:m].copy()).cuda()
        c, r = G.chi2(g, d, obs, want_resid=True)
        maps = G.eval_maps(g, d)
        jtj = torch.empty((m, 10, 10), dtype=torch.float64, device="cuda")
        jtv = torch.empty((m, 10), dtype=torch.float64, device="cuda")
        c2 = torch.empty(m, dtype=torch.float64, device="cuda")
        jac = torch.empty((m, 10, 2, ny, nx), dtype=torch.float32, device="cuda")
        G.gbk_jacobian(g, d, obs, free, cot[:m].contiguous(), jtj, jtv, c2, jac)
        got.append([t[:3].cpu().numpy() for t in (c, r, maps, jtj, jtv, c2, jac)])
    for other in got[1:]:
        for a, b in zip(got[0], other):
            np.testing.assert_array_equal(a.view(np.uint8), b.view(np.uint8))


def test_fits_agree(G):
    """A fit of 320 fields, whose running ones shrink through both kernels,
    and of its first eight alone."""
    rng = np.random.default_rng(9)
    nx, ny, n = 40, 36, 320
    g = Geometry(nx, ny, 1, 10.0, model=2)
    p = _params(nx, ny, n, rng)
    v = G.eval_maps(g, torch.from_numpy(p)).cpu().numpy()[:, 1]
    obs = [_obs(G, nx, ny, rng, v[i]) for i in range(n)]
    free = (0, 1, 2, 3, 4, 5, 6, 8, 9)
    lo, hi = p.copy(), p.copy()
    for k, (a, b) in {0: (0, nx - 1), 1: (0, ny - 1), 2: (-360, 720), 3: (1, 89), 4: (-200, 200), 5: (1, 600),
                      6: (0.05, 100), 8: (0.1, 5), 9: (0.05, 5)}.items():
        lo[:, k], hi[:, k] = a, b
    start = np.array([synth.perturb(rng, q, free, 0.1, lo[i], hi[i]) for i, q in enumerate(p)])
    o = G.lm_opts(max_iter=60, jacobian=G.JAC_TANGENT, free=free)
    whole = G.fit_lm(g, obs, start, lo, hi, o)
    part = G.fit_lm(g, obs[:8], start[:8], lo[:8], hi[:8], o)
    for a, b in zip(whole, part):
        np.testing.assert_array_equal(a[:8].view(np.uint8), b.view(np.uint8))
