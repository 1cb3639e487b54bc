"""The velocity-field sums over their chains of pixels (256 chains, eight
groups, eight steps at a time) at the sizes where a chain, a group or a block
of steps begins or ends: chi2 and the normal equations against FP64 sums of
the residual and Jacobian maps of the same call.

Tolerance: a chain of n / 256 + 1 FP32 terms and five levels of the sum over
32 chains round at most n / 256 + 6 times; with 2^-24 each, of the sum of the
terms' magnitudes."""
import numpy as np
import pytest
import torch

from paper_1510_01815_gb300.synth import Geometry

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model", [1, 2])
@pytest.mark.parametrize("nx,ny", [(1, 1), (31, 1), (32, 1), (33, 1), (256, 1), (257, 1), (2048, 1), (2049, 1), (91, 53)])
def test_chain_sums(nx, ny, model):
    from paper_1510_01815_gb300 import build, gbk as G
    build.build()
    rng = np.random.default_rng(nx + ny)
    g = Geometry(nx, ny, 1, 10.0, model=model)
    n = 3
    p = np.tile([0.4 * nx, 0.6 * ny, 30.0, 50.0, 5.0, 200.0, 4.0, 30.0, 1.2, 0.9], (n, 1))
    p[:, 2] = rng.uniform(0, 360, n)
    f = lambda a: torch.from_numpy(a.astype(np.float32)).cuda()
    obs = G.Obs(f(rng.normal(0, 80, (ny, nx))), f(rng.uniform(20, 40, (ny, nx))), f(rng.uniform(0.1, 0.3, (ny, nx))),
                f(rng.uniform(0.1, 0.3, (ny, nx))), torch.from_numpy((rng.uniform(size=(ny, nx)) > 0.1).astype(np.uint8)).cuda())
    d = torch.from_numpy(p).cuda()
    c, r = G.chi2(g, d, obs, want_resid=True)
    free = tuple(range(10))
    jtj = torch.empty((n, 10, 10), dtype=torch.float64, device="cuda")
    jtv = torch.empty((n, 10), dtype=torch.float64, device="cuda")
    c2 = torch.empty(n, dtype=torch.float64, device="cuda")
    jac = torch.empty((n, 10, 2, ny, nx), dtype=torch.float32, device="cuda")
    G.gbk_jacobian(g, d, obs, free, None, jtj, jtv, c2, jac)
    J = jac.cpu().double().numpy().reshape(n, 10, -1)
    R = r.cpu().double().numpy().reshape(n, -1)
    tol = (nx * ny / 256 + 6) * 2.0 ** -24
    for i in range(n):
        s = float((R[i] ** 2).sum())
        assert abs(float(c[i]) - s) <= 2 * tol * s
        # the Jacobian's residuals agree with the evaluator's to rounding
        assert abs(float(c2[i]) - s) <= 1e-5 * s + 1e-12
        np.testing.assert_array_less(np.abs(jtj[i].cpu().numpy() - J[i] @ J[i].T), tol * 2 * np.abs(J[i]) @ np.abs(J[i]).T + 1e-30)
        mag = np.abs(J[i]) @ np.abs(R[i])
        np.testing.assert_array_less(np.abs(jtv[i].cpu().numpy() - J[i] @ R[i]), 1e-5 * mag + 1e-30)
