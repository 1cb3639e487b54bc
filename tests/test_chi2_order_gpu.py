"""The sum of chi2 has one order whatever shape a call takes: the same bits in
batches of 1 to 2048 models (small batches of large images take the residuals
in a shape of their own and sum them in the large batch's order), with
residuals and without; its value against an FP64 sum of the call's own
residuals.

Tolerance: a thread's terms are compensated, 5 levels of FP32 sums follow; all
terms are positive, so 8 x 2^-24 of the sum bounds it."""
import numpy as np
import pytest
import torch

from paper_1510_01815_gb300 import synth
from paper_1510_01815_gb300.synth import Geometry

pytestmark = pytest.mark.gpu

# one CTA at every batch size, cut into tiles at some of them, and at all; rows
# and columns that leave the last task a remainder
SIZES = [(1, 1), (16, 16), (17, 33), (32, 32), (64, 63), (90, 77), (128, 128), (131, 15), (7, 200), (192, 192)]


@pytest.mark.parametrize("psf", [0.0, 2.5, 4.7])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_chi2_bits_and_value(nx, ny, psf):
    from paper_1510_01815_gb300 import build, gbk as G
    build.build()
    g = Geometry(nx, ny, 16, 30.0, 0.0, psf, 40.0)
    rng = np.random.default_rng(nx + ny)
    p = synth.draw_fp_params(rng, 2048 if nx * ny < 9000 else 300, g, 0.15 * max(nx, ny) + 1.0)
    p[2, synth.SIG0] = -1.0  # outside the parameter domain: NaN
    f = lambda a: torch.from_numpy(a.astype(np.float32)).cuda()
    shape = (ny, nx)
    obs = G.Obs(f(rng.normal(0, 80, shape)), f(rng.uniform(20, 40, shape)), f(rng.uniform(0.1, 0.3, shape)),
                f(rng.uniform(0.1, 0.3, shape)), torch.from_numpy((rng.uniform(size=shape) > 0.1).astype(np.uint8)).cuda())
    d = torch.from_numpy(p).cuda()
    ref, r = G.chi2(g, d[:5].contiguous(), obs, flags=G.PATH_SPLIT, want_resid=True)
    ref, r = ref.cpu().numpy(), r.cpu().double().numpy().reshape(5, -1)
    assert np.isnan(ref[2])
    for i in (0, 1, 3, 4):
        s = float((r[i] ** 2).sum())
        assert abs(ref[i] - s) <= 8 * 2.0 ** -24 * s
    for n in (3, 40, 130, 300, 2048):
        if n > len(p):
            continue
        got = G.chi2(g, d[:n].contiguous(), obs, flags=G.PATH_SPLIT).cpu().numpy()[:5]
        np.testing.assert_array_equal(got.view(np.uint64), ref[:len(got)].view(np.uint64))
