"""A non-finite observed pixel reaches the features of its own 2 x 2 patch
alone: the ReLU takes NaN for 0, so those 32 features are 0.  With negative
biases in the first layer a patch whose four pixels are masked has the same
features, so both maps must give the same outputs to the bit."""
import numpy as np
import pytest
import torch

from oracle import cnn
from test_cnn_gpu import _dev, _problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("which", ["v", "s"])
@pytest.mark.parametrize("B", [8, 160])
def test_nan_stays_in_its_patch(B, which):
    from paper_1510_01815_gb300 import build, gbk as G
    build.build()
    P, v, s, mask, _ = _problem(70 + B, B)
    first = P[:cnn.C[0] * (cnn.K[0] + 1)].reshape(cnn.C[0], cnn.K[0] + 1)
    first[:, -1] = -np.abs(first[:, -1]) - 1e-3
    mask[:] = 1
    masked, bad = mask.copy(), {"v": v.copy(), "s": s.copy()}
    # one patch in each position of a group of four (in Morton order, a 4 x 4
    # block of pixels), a pair in one group, and corners of the map
    for b, Y, X in [(0, 0, 0), (0, 5, 6), (1, 8, 9), (2, 9, 8), (3, 11, 11), (4, 20, 20), (4, 20, 21), (5, 31, 31),
                    (B - 1, 31, 0)]:
        masked[b, 2 * Y:2 * Y + 2, 2 * X:2 * X + 2] = 0
        bad[which][b, 2 * Y + (b & 1), 2 * X + (b >> 1 & 1)] = np.nan
    outs = []
    for vv, ss, mm in ((bad["v"], bad["s"], mask), (v, s, masked), (v, s, mask)):
        dP, dv, ds, dm = _dev(P.astype(np.float32), vv, ss, mm)
        ws = torch.empty(G.gbk_cnn_workspace_bytes(B), dtype=torch.uint8, device="cuda")
        out = torch.empty((B, 16), dtype=torch.float32, device="cuda")
        G.gbk_cnn_forward(dP, dv, ds, dm, out, ws)
        outs.append(out.cpu().numpy())
    assert np.isfinite(outs[0]).all()
    np.testing.assert_array_equal(outs[0].view(np.uint32), outs[1].view(np.uint32))
    # the maps without a bad pixel are untouched, the others are not
    same = (outs[0] == outs[2]).all(axis=1)
    assert list(np.flatnonzero(~same)) == sorted({0, 1, 2, 3, 4, 5, B - 1})
