"""Model cubes in one kernel (u = 1, small radii): against the FP64 oracle,
against the moments of a chi2 call (residuals from zero maps of unit weight),
and a model alone (channels cut into ranges, moments
from the cube) against the same model in a batch that fills the chip (not
cut): the same terms in the same order, so the same bits.

Tolerances: a voxel's Gaussian carries the FP32 error of its exponent (|log2|
up to 150 at 2^-23, times ln 2: 1.3e-5 where it is smallest, 2e-6 above a
tenth of the peak), the PSF and LSF passes some 45 roundings; 1e-5 of the
cube's peak.  The moments of the two calls: 2e-5 of the scale of a map, the
larger of |m1| and V_max, of m2 and sigma0."""
import numpy as np
import pytest
import torch

import oracle
from cases import ogeom
from paper_1510_01815_gb300 import synth
from paper_1510_01815_gb300.synth import Geometry

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 340])  # channels cut into ranges, and not
@pytest.mark.parametrize("nx,ny,nz,psf,lsf", [
    (1, 1, 1, 0.0, 0.0),      # radii 0
    (64, 16, 7, 0.5, 20.0),   # one tile exactly; a batch of channels exactly or nearly
    (65, 17, 13, 2.3, 40.0),  # a tile and a remainder of one
    (30, 41, 33, 3.0, 60.0),  # odd radii, rows without 16-byte stores
    (12, 8, 40, 4.6, 70.0),   # the largest radii
    (12, 8, 40, 4.6, 92.0),   # an LSF beyond them: the chain
])
def test_cube_kernel(nx, ny, nz, psf, lsf, n):
    from paper_1510_01815_gb300 import build, gbk
    build.build()
    g = Geometry(nx, ny, nz, 20.0, 5.0, psf, lsf)
    rng = np.random.default_rng(5)
    ps = np.array([synth.params(rng.uniform(0.4, 0.6) * nx, rng.uniform(0.4, 0.6) * ny, rng.uniform(0, 360),
                                rng.uniform(30, 75), 4.0, 8.0 * nz, 2.0, rng.uniform(12, 60), 1.3, 0.2 * nx + 1)
                   for _ in range(n)])
    if n > 1:
        ps[1, synth.INCL] = 95.0  # outside the domain: NaN throughout
    par = torch.from_numpy(ps).cuda()
    cubes, maps = gbk.eval_cubes(g, par)
    zero = np.zeros((ny, nx), np.float32)
    obs = gbk.Obs.from_numpy(zero, zero, zero + 1, zero + 1, np.ones((ny, nx), np.uint8))
    _, resid = gbk.chi2(g, par, obs, flags=gbk.PATH_STAGED, want_resid=True)
    if n > 1:
        assert torch.isnan(cubes[1]).all() and torch.isnan(maps[1]).all()
    keep = [i for i in range(n) if i != 1]
    valid = maps[keep, 0] > 0
    for k, floor in ((1, synth.VMAX), (2, synth.SIG0)):
        scale = torch.maximum(maps[keep, k].abs(), torch.from_numpy(ps[keep, floor]).float().cuda()[:, None, None])
        assert ((maps[keep, k] - resid[keep, k - 1]).abs() / scale)[valid].max() <= 2e-5
    assert (resid[keep][:, 0][~valid] == 0).all()
    for i in (0, n - 1):
        if i == 1:
            continue
        ref, _ = oracle.evaluate(ogeom(g), ps[i], want_cube=True)
        assert np.abs(cubes[i].cpu().numpy() - ref).max() <= 1e-5 * np.abs(ref).max()
    only = torch.empty_like(cubes)  # without the maps
    gbk.gbk_eval_cubes(g, par, cubes=only, workspace=gbk.workspace_for(g, n, gbk.PATH_STAGED, "cuda"))
    assert torch.equal(torch.nan_to_num(only, -1.0), torch.nan_to_num(cubes, -1.0))
    c1, m1 = gbk.eval_cubes(g, par[:1])
    assert torch.equal(c1[0], cubes[0]) and torch.equal(m1[0], maps[0])
