"""The CNN's forward pass and gradient at batch sizes that take the dense
layers' products through their different tiles (a single row of tiles, narrow
tiles, the four-part transposed copies, several CTAs per SM), element by
element against the oracle's BF16 form with the tolerance of test_cnn_gpu."""
import pytest
import torch

from oracle import cnn
from test_cnn_gpu import _assert_close_elementwise, _dev, _problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [8, 24, 160, 312])
def test_batch_sizes(B):
    from paper_1510_01815_gb300 import build, gbk as G
    build.build()
    P, v, s, mask, t = _problem(40 + B, B)
    dP, dv, ds, dm, dt = _dev(P.astype("float32"), v, s, mask, t)
    ws = torch.empty(G.gbk_cnn_workspace_bytes(B), dtype=torch.uint8, device="cuda")
    out = torch.empty((B, 16), dtype=torch.float32, device="cuda")
    G.gbk_cnn_forward(dP, dv, ds, dm, out, ws)
    x = cnn.encode(v, s, mask, rounding="bf16")
    _assert_close_elementwise(out.cpu().numpy(), cnn.forward(P, x, rounding="bf16")[0], "forward output")
    grad = torch.empty(cnn.param_count(), dtype=torch.float32, device="cuda")
    loss = torch.empty(1, dtype=torch.float32, device="cuda")
    G.gbk_cnn_grad(dP, dv, ds, dm, dt, grad, loss, ws)
    ref_loss, ref_g = cnn.loss_and_grad(P, x, t.astype("float64"), rounding="bf16")
    assert abs(float(loss) - ref_loss) <= 2e-3 * ref_loss
    g, off = grad.cpu().numpy(), cnn.param_offsets()
    for l in range(cnn.NL):
        W = g[off[l]:off[l + 1]].reshape(cnn.C[l], cnn.K[l] + 1)
        R = ref_g[off[l]:off[l + 1]].reshape(cnn.C[l], cnn.K[l] + 1)
        _assert_close_elementwise(W[:, :-1], R[:, :-1], "layer %d weight gradient" % l)
        _assert_close_elementwise(W[:, -1], R[:, -1], "layer %d bias gradient" % l)
    assert G.gbk_device_status() == 0
