"""The split path's line sums (closed form, polynomials at the band edges,
direct sum) against the FP64 oracle, at the line widths and velocities where
one form hands over to the next, and at the edges of its tiles.

Tolerance: the interpolation error of the forms is below 2e-7 of the sums; the
sums and the two 2R + 1 tap filters add FP32 roundings of up to some 230 terms,
sqrt(230) 2^-24 = 9e-7; the moments combine three such sums.  Twenty times that
is 2e-5 of the scale of each map (m0: its maximum; m1: the larger of |m1| and
V_max; m2: the larger of m2 and sigma0).  A line centred a distance d beyond
the band is seen by its Gaussian tail alone, whose logarithm has the slope
d / s^2 in the line's velocity: FP32 velocities (a few roundings of the
largest one, 4 x 2^-24 |v|) move all its sums by that factor, which is the
same for any way of summing them and is added."""
import numpy as np
import pytest
import torch

import oracle
from cases import make_obs, ogeom
from paper_1510_01815_gb300 import synth
from paper_1510_01815_gb300.synth import Geometry

pytestmark = pytest.mark.gpu

TOL = 2e-5


@pytest.fixture(scope="module")
def G():
    from paper_1510_01815_gb300 import build, gbk
    build.build()
    assert torch.cuda.is_available()
    return gbk


def _params(g, sig, vmax, n=3):
    rng = np.random.default_rng(17)
    out = []
    for k in range(n):
        out.append(synth.params(rng.uniform(0.4, 0.6) * g.nx, rng.uniform(0.4, 0.6) * g.ny, rng.uniform(0, 360),
                                rng.uniform(30, 75), rng.uniform(-10, 10), vmax * (1 if k else -1), rng.uniform(1, 4),
                                sig, rng.uniform(0.5, 2.0), 0.15 * max(g.nx, g.ny) + 1.0))
    return np.array(out)


def _check(g, got, ref, ps):
    for i in range(len(ps)):
        vmax = abs(ps[i, synth.VMAX]) * np.sin(np.radians(ps[i, synth.INCL])) + abs(ps[i, synth.VSYS])
        beyond = max(0.0, vmax + abs(g.vc) - 0.5 * (g.nz - 1) * g.dv)
        tol = TOL + 4 * 2.0 ** -24 * vmax * beyond / ps[i, synth.SIG0] ** 2
        ok = (ref[i, 0] > 1e-18 * ps[i, synth.I0]) & (got[i, 0] > 0)  # away from the invalid-spectrum threshold
        scale = (np.full_like(ref[i, 0], ref[i, 0].max()), np.maximum(np.abs(ref[i, 1]), abs(ps[i, synth.VMAX])),
                 np.maximum(ref[i, 2], ps[i, synth.SIG0]))
        for k in range(3):
            err = (np.abs(got[i, k] - ref[i, k]) / scale[k])[ok]
            assert err.size == 0 or err.max() <= tol, (i, k, err.max(), tol)


# line widths in channels around the hand-overs (0.25: narrowest polynomial,
# 0.45: narrowest closed form, 1.15: no ripple left), and velocity ranges
# inside the band, up to its edges and far beyond them
@pytest.mark.parametrize("lsf_mode,lsf", [(0, 30.0), (1, 20.0), (0, 0.0)])
@pytest.mark.parametrize("width", [0.2, 0.26, 0.44, 0.46, 0.8, 1.14, 1.16, 4.0])
@pytest.mark.parametrize("reach", [0.3, 1.0, 2.0])
def test_line_forms_vs_oracle(G, width, reach, lsf_mode, lsf):
    g = Geometry(21, 18, 24, 20.0, 3.0, 2.0, lsf, lsf_mode)
    sig = width * g.dv
    if lsf_mode == 1:  # the width the line ends up with
        sig = np.sqrt(max(sig ** 2 - (lsf / 2.3548200450309493) ** 2, 1.0))
    ps = _params(g, sig, reach * 0.5 * g.nz * g.dv)
    ref = oracle.evaluate_batch(ogeom(g), ps)
    got = G.eval_maps(g, torch.from_numpy(ps), split=True).cpu().numpy().astype(np.float64)
    _check(g, got, ref, ps)


# image sizes at the edges of the tasks (pairs, fours) and of the tiles; PSF
# radii 0, odd and the largest
@pytest.mark.parametrize("nx,ny", [(1, 1), (2, 3), (4, 4), (5, 2), (7, 66), (67, 9), (83, 85), (130, 6)])
@pytest.mark.parametrize("psf", [0.0, 0.5, 1.7, 4.7])
def test_tile_edges_vs_oracle(G, nx, ny, psf):
    g = Geometry(nx, ny, 12, 30.0, 0.0, psf, 40.0)
    ps = _params(g, 45.0, 120.0, n=2)
    ref = oracle.evaluate_batch(ogeom(g), ps)
    got = G.eval_maps(g, torch.from_numpy(ps), split=True).cpu().numpy().astype(np.float64)
    _check(g, got, ref, ps)


@pytest.mark.parametrize("g", [synth.SINGLE_GEOM, Geometry(96, 70, 32, 20.0, 0.0, 3.0, 30.0)])
def test_chi2_does_not_depend_on_the_batch(G, g):
    """A model's chi2 is the same to the bit in batches of any size."""
    ps = _params(g, 40.0, 180.0, n=1).repeat(300, axis=0)
    obs = make_obs(g, ps[0], seed=3)
    d = G.Obs.from_numpy(obs.v, obs.s, obs.w_v, obs.w_s, obs.mask)
    got = [G.chi2(g, torch.from_numpy(ps[:n]), d, flags=G.PATH_SPLIT).cpu().numpy() for n in (1, 7, 300)]
    assert len(set(np.concatenate(got))) == 1
