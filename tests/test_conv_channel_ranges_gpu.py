"""The staged convolution for wide PSFs cuts a tile's channels into ranges when
the tiles alone do not fill the chip.  Every output channel takes the same
terms in the same order either way, so one model alone (cut) gives the same
bits as the same model in a batch that fills the chip (not cut)."""
import pytest
import torch

from paper_1510_01815_gb300 import synth
from paper_1510_01815_gb300.synth import Geometry

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,fwhm", [
    (33, 31, 40, 8.3),   # odd rows (scalar stores), tiles with a one-column remainder
    (32, 32, 17, 9.0),   # one tile, a short band
    (64, 34, 9, 11.5),   # channels fewer than the ranges that are tried
])
def test_ranges_do_not_change_bits(nx, ny, nz, fwhm):
    from paper_1510_01815_gb300 import build, gbk
    build.build()
    g = Geometry(nx, ny, nz, 20.0, psf_fwhm=fwhm, lsf_fwhm=46.0)
    p = synth.params(0.47 * nx, 0.52 * ny, 33.0, 51.0, 12.0, 180.0, 3.0, 35.0, 1.0, 0.2 * nx)
    one = torch.from_numpy(p[None])
    n = 912  # whole waves of tiles on 152 SMs, one or two tiles each
    cubes1, maps1 = gbk.eval_cubes(g, one)
    cubes, maps = gbk.eval_cubes(g, one.repeat(n, 1))
    for i in (0, n // 2, n - 1):
        assert torch.equal(cubes1[0], cubes[i])
        assert torch.equal(maps1[0], maps[i])
