"""A model's maps are the same to the bit in batches of any size (the tiles
that an image is cut into depend on the batch), whichever form its lines take:
closed, polynomials at the band's edges, or the direct sum that single lanes
of a warp fall back to."""
import numpy as np
import pytest
import torch

from paper_1510_01815_gb300 import synth
from paper_1510_01815_gb300.synth import Geometry

pytestmark = pytest.mark.gpu

BASE = Geometry(96, 80, 40, 15.0, 0.0, 3.0, 30.0)
CASES = {
    "inside the band": (BASE, {}),
    "narrow line": (BASE.with_(dv=60.0, lsf_fwhm=0.0), {synth.SIG0: 10.0}),
    "beyond the band": (BASE.with_(nz=12), {synth.VMAX: 600.0}),
    "narrow line beyond the band": (BASE.with_(nz=12, dv=30.0), {synth.SIG0: 6.0, synth.VMAX: 600.0}),
    "narrow band": (BASE.with_(nz=8, dv=10.0), {}),
    "one channel": (BASE.with_(nz=1), {}),
    "small image": (Geometry(9, 7, 30, 20.0, 0.0, 2.5, 30.0), {}),
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_maps_do_not_depend_on_the_batch(case):
    from paper_1510_01815_gb300 import build, gbk as G
    build.build()
    g, over = CASES[case]
    p = synth.draw_fp_params(np.random.default_rng(3), 2048, g, 0.1 * g.nx)
    for k, v in over.items():
        p[:, k] = v
    d = torch.from_numpy(p).cuda()
    ref = None
    for n in (1, 7, 64, 500, 2048):
        maps = torch.empty((n, 3, g.ny, g.nx), dtype=torch.float32, device="cuda")
        G.gbk_eval_cubes(g, d[:n].contiguous(), maps=maps, workspace=G.workspace_for(g, n, G.PATH_SPLIT, "cuda"))
        first = maps[0].cpu().numpy().view(np.uint32)
        ref = first if ref is None else ref
        np.testing.assert_array_equal(first, ref)
