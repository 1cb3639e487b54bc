"""The work this framework is used for, as measurable cases.

Every case is one call (or one training step) through the package's public
entry points, at sizes taken from the repository's own workloads: the single
galaxy (32 x 32 x 64), the Fabry-Perot galaxy (192 x 192 x 48), the nested
grid (64^3), the survey of uneven cubes, the learned seed's 64 x 64 maps and
the 256 x 256 velocity fields.  `exact` restates each model in 64-bit torch.
"""
import math

import numpy as np
import torch

from paper_1510_01815_gb300 import gbk, synth

FWHM = 2.0 * math.sqrt(2.0 * math.log(2.0))
CNN_C = (32, 64, 128, 256, 256, 16)
CNN_K = (16, 128, 256, 512, 4096, 256)
LR = 1e-3


def listed():
    single = dict(nx=32, ny=32, nz=64, dv=20.0, psf=2.5, lsf=30.0, mode=0, up=1)
    grid = dict(single, nx=64, ny=64)
    return [
        # one model of a small galaxy: a caller's own optimiser asking for one model at a time
        dict(name="maps-single-1", kind="maps", n=1, **single),
        # one iteration's models of a batch of small galaxies (a batched fit, a V_t - i degeneracy map)
        dict(name="maps-single-2048", kind="maps", n=2048, **single),
        # the live points of nested sampling on a Fabry-Perot galaxy: one launch per iteration
        dict(name="maps-fabry-perot-400", kind="maps", n=400, nx=192, ny=192, nz=48, dv=10.0, psf=3.0, lsf=30.0,
             mode=0, up=1),
        # a chunk of a nested grid's nodes, or of the learned seed's training set: the largest batch
        dict(name="maps-grid-8192", kind="maps", n=8192, **grid),
        # the same maps by the one-line call, which allocates its output and keeps no workspace; a ragged
        # rectangle, an odd channel count, the LSF folded into the line width
        dict(name="eval-maps-odd-77", kind="eval", n=77, nx=57, ny=43, nz=37, dv=15.0, psf=3.5, lsf=35.0, mode=1,
             up=1),
        # a trial model of each galaxy of a survey of uneven cubes (24 - 96 spaxels, 32 - 128 channels)
        dict(name="survey-2048", kind="survey", n=2048),
        # materialised model cubes (for plots, residual cubes, mock data)
        dict(name="cubes-grid-256", kind="cubes", n=256, **grid),
        # cubes modelled on a grid twice as fine and averaged down (Sec. 2.2.4)
        dict(name="cubes-upsampled-32", kind="cubes", n=32, **dict(single, up=2)),
        # Jacobian maps of the residuals (all ten parameters): error analysis, a caller's own optimiser
        dict(name="jacobian-256", kind="jacobian", n=256, **single),
        # the learned seed's prediction for a batch of galaxies
        dict(name="seed-forward-1024", kind="forward", n=1024),
        # one training step of the learned seed
        dict(name="seed-train-1024", kind="train", n=1024),
        # a whole fit: nine-parameter velocity fields with the Epinat curve, analytic Jacobian
        dict(name="fit-fields-64", kind="fit", n=64, nx=256, ny=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["maps", "maps", "maps", "eval", "survey", "cubes", "jacobian", "forward", "train", "fit"])
    if kind == "survey":
        return dict(kind=kind, n=_log_int(rng, 16, 2048))
    if kind in ("forward", "train"):  # batches are multiples of 8
        return dict(kind=kind, n=8 * _log_int(rng, 2, 128))
    if kind == "fit":
        return dict(kind=kind, n=_log_int(rng, 2, 64), nx=_log_int(rng, 48, 256), ny=_log_int(rng, 48, 256))
    small = kind == "jacobian"  # its widest served maps are near 100 x 100 spaxels
    nx, ny = _log_int(rng, 24, 64 if small else 192), _log_int(rng, 24, 64 if small else 192)
    nz = _log_int(rng, 32, 128)
    up = rng.choice([1, 1, 2]) if kind == "cubes" else 1
    most = {"maps": 2.1e9, "eval": 2.5e8, "cubes": 6.7e7 if up == 1 else 2.1e6, "jacobian": 1.6e7}[kind]  # voxels
    n = _log_int(rng, 1, max(1, min(8192, int(most / (nx * ny * nz)))))
    return dict(kind=kind, n=n, nx=nx, ny=ny, nz=nz, dv=float(rng.choice([10.0, 15.0, 20.0])),
                psf=round(rng.uniform(1.5, 3.9), 2), lsf=round(rng.uniform(20.0, 60.0), 1),
                mode=rng.choice([0, 0, 1]), up=up)


# ----------------------------------------------------------------------------
# Inputs, from the seed alone.
def _geom(case):
    return synth.Geometry(case["nx"], case["ny"], case["nz"], case["dv"], 0.0, case["psf"], case["lsf"],
                          case["mode"], case["up"])


def _disc_params(case, seed):
    """Parameter sets over the Fabry-Perot ranges, centre in 0.4 - 0.6 of the
    frame, scale length a tenth of it or so."""
    rng = np.random.default_rng([seed, 1])
    n, size = case["n"], min(case["nx"], case["ny"])
    p = np.zeros((n, 10))
    p[:, 0] = rng.uniform(0.4, 0.6, n) * case["nx"]
    p[:, 1] = rng.uniform(0.4, 0.6, n) * case["ny"]
    p[:, 2] = rng.uniform(0.0, 360.0, n)
    p[:, 3] = rng.uniform(20.0, 80.0, n)
    p[:, 4] = rng.uniform(-20.0, 20.0, n)
    p[:, 5] = rng.uniform(50.0, 300.0, n)
    p[:, 6] = rng.uniform(1.0, 8.0, n)
    p[:, 7] = rng.uniform(10.0, 80.0, n)
    p[:, 8] = 1.0
    p[:, 9] = rng.uniform(0.09, 0.14, n) * size
    return p


def _weights(case, seed, dev):
    """Weights of 5 km/s errors and a mask of 2 % dead fibres."""
    rng = np.random.default_rng([seed, 2])
    shape = (case["ny"], case["nx"])
    wv = torch.full(shape, 1.0 / 5.0, dtype=torch.float32, device=dev)
    ws = torch.full(shape, 1.0 / (5.0 * math.sqrt(2.0)), dtype=torch.float32, device=dev)
    mask = torch.from_numpy((rng.uniform(size=shape) >= 0.02).astype(np.uint8)).to(dev)
    return wv, ws, mask


def _field(nx, ny, p, dev, epinat):
    """Velocity fields [n][ny][nx] in 64 bits (Eqs. 1-4, 6, 7 and 8)."""
    p = torch.as_tensor(p, dtype=torch.float64, device=dev)
    c = [p[:, k].reshape(-1, 1, 1) for k in range(10)]
    x = torch.arange(nx, dtype=torch.float64, device=dev).reshape(1, 1, nx)
    y = torch.arange(ny, dtype=torch.float64, device=dev).reshape(1, ny, 1)
    pa, inc = torch.deg2rad(c[2]), torch.deg2rad(c[3])
    xe = -(x - c[0]) * torch.sin(pa) + (y - c[1]) * torch.cos(pa)
    ye = (-(x - c[0]) * torch.cos(pa) - (y - c[1]) * torch.sin(pa)) / torch.cos(inc)
    r = torch.sqrt(xe * xe + ye * ye)
    if epinat:
        v = c[5] * (r / c[6]) ** c[9] / (1.0 + (r / c[6]) ** c[8])
    else:
        v = 2.0 / math.pi * c[5] * torch.atan(r / c[6])
    return c[4] + v * xe / torch.clamp(r, min=1e-30) * torch.sin(inc)


def _seed_data(n, seed, dev):
    """Observed 64 x 64 maps, targets, and a network in mid-training."""
    rng = np.random.default_rng([seed, 3])
    p = synth.draw_cnn_params(rng, n)
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed) * 7919 + 11)
    v = torch.empty((n, 64, 64), dtype=torch.float32, device=dev)
    for i in range(0, n, 256):
        v[i:i + 256] = _field(64, 64, p[i:i + 256], dev, False).float()
    v += 5.0 * torch.randn(v.shape, generator=g, device=dev)
    sig = torch.as_tensor(p[:, 7], dtype=torch.float32, device=dev).reshape(-1, 1, 1).expand(n, 64, 64).contiguous()
    sig += 5.0 * math.sqrt(2.0) * torch.randn(sig.shape, generator=g, device=dev)
    mask = (torch.rand(v.shape, generator=g, device=dev) >= 0.02).to(torch.uint8)
    pa = np.radians(p[:, 2])
    t = np.stack([(p[:, 0] - 31.5) / 8, (p[:, 1] - 31.5) / 8, np.cos(pa), np.sin(pa), (p[:, 3] - 50) / 20,
                  p[:, 4] / 30, (p[:, 5] - 175) / 75, (p[:, 6] - 4.5) / 2.5, (p[:, 7] - 45) / 25,
                  (p[:, 9] - 7) / 3], axis=1)
    blocks = []
    for c, k in zip(CNN_C, CNN_K):
        b = torch.randn((c, k + 1), generator=g, device=dev) * math.sqrt(2.0 / k)
        b[:, k] *= 0.1
        blocks.append(b.reshape(-1))
    w = torch.cat(blocks)
    m = 1e-3 * torch.randn(w.shape, generator=g, device=dev)
    u = 1e-6 * (0.5 + torch.rand(w.shape, generator=g, device=dev))
    return v, sig, mask, torch.as_tensor(t, dtype=torch.float32, device=dev), w, m, u


def _fit_problem(case, seed, dev):
    """Noisy Epinat fields, starts 10 % off the truth, and the fit's bounds."""
    rng = np.random.default_rng([seed, 4])
    n, nx, ny = case["n"], case["nx"], case["ny"]
    p = np.zeros((n, 10))
    p[:, 0], p[:, 1] = rng.uniform(0.45, 0.55, n) * nx, rng.uniform(0.45, 0.55, n) * ny
    p[:, 2], p[:, 3], p[:, 4] = rng.uniform(0, 360, n), rng.uniform(30, 70, n), rng.uniform(-50, 50, n)
    p[:, 5], p[:, 6] = rng.uniform(100, 300, n), rng.uniform(0.02, 0.12, n) * min(nx, ny)
    p[:, 7], p[:, 8], p[:, 9] = 30.0, rng.uniform(0.6, 2.5, n), rng.uniform(0.5, 1.5, n)
    lo, hi = p.copy(), p.copy()
    for k, (a, b) in {0: (0, nx - 1), 1: (0, ny - 1), 2: (-360, 720), 3: (1, 89), 4: (-200, 200), 5: (1, 600),
                      6: (0.05, 100), 8: (0.1, 5), 9: (0.05, 5)}.items():
        lo[:, k], hi[:, k] = a, b
    free = (0, 1, 2, 3, 4, 5, 6, 8, 9)
    start = np.array([synth.perturb(rng, p[i], free, 0.1, lo[i], hi[i]) for i in range(n)])
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed) * 7919 + 13)
    v = torch.cat([_field(nx, ny, p[i:i + 16], dev, True) for i in range(0, n, 16)]).float()
    v += 5.0 * torch.randn(v.shape, generator=g, device=dev)
    return v, start, lo, hi, free


def _survey(n, seed):
    """The survey's galaxies, and a trial's parameter sets around theirs."""
    drawn = synth.draw_survey(np.random.default_rng(n), n)
    rng = np.random.default_rng([seed, 5])
    lo, hi = np.full(10, -np.inf), np.full(10, np.inf)
    hi[3] = 88.0
    return [g for g, _ in drawn], np.array([synth.perturb(rng, p, frac=0.1, lo=lo, hi=hi) for _, p in drawn])


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def prepare(case, seed):
    dev, kind, n = _device(), case["kind"], case["n"]
    s = {"kind": kind}
    if kind in ("maps", "eval", "cubes", "jacobian"):
        g = s["geom"] = _geom(case)
        s["params"] = torch.from_numpy(_disc_params(case, seed)).to(dev)
        if kind in ("maps", "cubes"):
            s["maps"] = torch.empty((n, 3, g.ny, g.nx), dtype=torch.float32, device=dev)
            s["workspace"] = gbk.workspace_for(g, n, gbk.PATH_SPLIT if kind == "maps" else gbk.PATH_STAGED, dev)
        if kind == "cubes":
            s["cubes"] = torch.empty((n, g.nz, g.ny, g.nx), dtype=torch.float32, device=dev)
        if kind == "jacobian":
            wv, ws, mask = _weights(case, seed, dev)
            field = _field(g.nx, g.ny, _disc_params(dict(case, n=1), seed), dev, False)[0].float().contiguous()
            s["obs"] = gbk.Obs(field, torch.full_like(field, 45.0), wv, ws, mask)
            s["jac"] = torch.empty((n, 10, 2, g.ny, g.nx), dtype=torch.float32, device=dev)
    elif kind == "survey":
        geoms, params = _survey(n, seed)
        s["geoms"] = gbk.cgeoms(geoms)
        s["params"] = torch.from_numpy(params).to(dev)
        s["maps"] = torch.empty(3 * gbk.survey_pix_offsets(geoms)[-1], dtype=torch.float32, device=dev)
        s["workspace"] = torch.empty(gbk.gbk_survey_workspace_bytes(geoms), dtype=torch.uint8, device=dev)
    elif kind in ("forward", "train"):
        v, sig, mask, t, w, m, u = _seed_data(n, seed, dev)
        s.update(v=v, sigma=sig, mask=mask, targets=t, weights=w, adam_m=m, adam_v=u, step=1000,
                 out=torch.empty((n, 16), dtype=torch.float32, device=dev),
                 loss=torch.empty(1, dtype=torch.float32, device=dev),
                 workspace=torch.empty(gbk.gbk_cnn_workspace_bytes(n), dtype=torch.uint8, device=dev))
    else:
        v, start, lo, hi, free = _fit_problem(case, seed, dev)
        s["geom"] = synth.Geometry(case["nx"], case["ny"], 1, 10.0, model=gbk.MODEL_VFIELD_EPINAT)
        shape = (case["ny"], case["nx"])
        sig = torch.full(shape, 30.0, dtype=torch.float32, device=dev)
        wv = torch.full(shape, 0.2, dtype=torch.float32, device=dev)
        ws = torch.zeros(shape, dtype=torch.float32, device=dev)  # velocity only
        ones = torch.ones(shape, dtype=torch.uint8, device=dev)
        s["obs"], s["keep"] = gbk.obs_array([gbk.Obs(v[i], sig, wv, ws, ones) for i in range(n)], dev)
        s["opts"] = gbk.lm_opts(max_iter=200, jacobian=gbk.JAC_TANGENT, free=free)
        s["start"], s["lo"], s["hi"] = (torch.from_numpy(a).to(dev) for a in (start, lo, hi))
        s["workspace"] = torch.empty(max(1, gbk.gbk_fit_lm_workspace_bytes(s["geom"], n, s["opts"])),
                                     dtype=torch.uint8, device=dev)
    return s


def run(s):
    kind = s["kind"]
    if kind == "maps":
        gbk.gbk_eval_cubes(s["geom"], s["params"], maps=s["maps"], workspace=s["workspace"])
        return {"maps": s["maps"]}
    if kind == "eval":
        return {"maps": gbk.eval_maps(s["geom"], s["params"])}
    if kind == "survey":
        gbk.gbk_survey_eval(s["geoms"], s["params"], maps=s["maps"], workspace=s["workspace"])
        return {"maps": s["maps"]}
    if kind == "cubes":
        gbk.gbk_eval_cubes(s["geom"], s["params"], cubes=s["cubes"], maps=s["maps"], workspace=s["workspace"])
        return {"cubes": s["cubes"], "maps": s["maps"]}
    if kind == "jacobian":
        gbk.gbk_jacobian(s["geom"], s["params"], s["obs"], tuple(range(10)), jac=s["jac"])
        return {"jac": s["jac"]}
    if kind == "forward":
        gbk.gbk_cnn_forward(s["weights"], s["v"], s["sigma"], s["mask"], s["out"], s["workspace"])
        return {"out": s["out"]}
    if kind == "train":
        s["step"] += 1
        gbk.gbk_cnn_train_step(s["weights"], s["adam_m"], s["adam_v"], s["step"], LR, s["v"], s["sigma"], s["mask"],
                               s["targets"], s["loss"], s["workspace"])
        return {"weights": s["weights"], "adam_m": s["adam_m"], "adam_v": s["adam_v"], "loss": s["loss"]}
    n, dev = s["start"].shape[0], s["start"].device
    p = s["start"].clone()  # fitted in place
    chi2 = torch.empty(n, dtype=torch.float64, device=dev)
    iters, status = (torch.empty(n, dtype=torch.int32, device=dev) for _ in range(2))
    gbk.gbk_fit_lm(s["geom"], s["obs"], s["lo"], s["hi"], p, s["opts"], chi2, iters, status, s["workspace"])
    return {"params": p, "chi2": chi2, "iters": iters, "status": status}


# ----------------------------------------------------------------------------
def _radius(fwhm_px):
    return math.ceil(4.0 * fwhm_px / FWHM) if fwhm_px > 0 else 0


def _map_flops(nx, ny, psf):
    """A spaxel's geometry, line moments (about 60 operations on the grid
    extended by the PSF's radius), two PSF passes on three moment sums and
    the quotients."""
    R = _radius(psf)
    ex, ey = nx + 2 * R, ny + 2 * R
    return 60.0 * ex * ey + 6.0 * (2 * R + 1) * (ey * nx + ny * nx) + 10.0 * nx * ny


def work(case):
    kind, n = case["kind"], case["n"]
    if kind in ("maps", "eval", "cubes", "jacobian"):
        nx, ny, nz, u = case["nx"], case["ny"], case["nz"], case["up"]
        b, f = 80.0 + 12.0 * nx * ny, _map_flops(u * nx, u * ny, u * case["psf"])
        if kind == "cubes":
            R, Rz = _radius(u * case["psf"]), _radius(u * case["lsf"] / case["dv"]) if case["mode"] == 0 else 0
            ex, ey, ez = u * nx + 2 * R, u * ny + 2 * R, u * nz + 2 * Rz
            vox = u ** 3 * nx * ny * nz
            b += 4.0 * nx * ny * nz
            f = 6.0 * ex * ey * ez + 2.0 * (2 * R + 1) * (ez * ey * u * nx + ez * u * u * nx * ny) \
                + 2.0 * (2 * Rz + 1) * vox + 5.0 * nx * ny * nz
        if kind == "jacobian":
            b, f = 80.0 + 80.0 * nx * ny, 11.0 * f
        return {"bytes": n * b + (9.0 * nx * ny if kind == "jacobian" else 0.0), "flops": n * f}
    if kind == "survey":  # the sizes' log-uniform means
        px = (96.0 ** 2 - 24.0 ** 2) / (2.0 * math.log(4.0))
        return {"bytes": n * (80.0 + 12.0 * px), "flops": n * _map_flops(math.sqrt(px), math.sqrt(px), 4.0)}
    if kind in ("forward", "train"):
        rows = (1024, 256, 64, 16, 1, 1)
        mac = sum(r * c * k for r, c, k in zip(rows, CNN_C, CNN_K))
        w = sum(c * (k + 1) for c, k in zip(CNN_C, CNN_K))
        if kind == "forward":
            return {"bytes": n * (9.0 * 4096 + 64) + 4.0 * w, "flops": 2.0 * n * mac}
        return {"bytes": n * (9.0 * 4096 + 40) + 24.0 * w, "flops": 2.0 * n * (3.0 * mac - rows[0] * CNN_C[0] * CNN_K[0])}
    px = float(case["nx"] * case["ny"])  # about ten iterations, each a Jacobian and a trial
    return {"bytes": n * (4.0 * px + 320.0) + 13.0 * px, "flops": n * px * 10.0 * (40.0 + 40.0 + 110.0)}


# ----------------------------------------------------------------------------
# The models in 64 bits.
def _taps(sigma, R, dev):
    if R == 0:
        return torch.ones(1, dtype=torch.float64, device=dev)
    j = torch.arange(-R, R + 1, dtype=torch.float64, device=dev)
    w = torch.exp(-0.5 * (j / sigma) ** 2)
    return w / w.sum()


def _band(taps, n):
    """[n][n + 2R]: the valid convolution with the taps as a matrix."""
    m = torch.zeros((n, n + len(taps) - 1), dtype=torch.float64, device=taps.device)
    for j in range(len(taps)):
        m.diagonal(j).copy_(taps[j].expand(n))
    return m


def _model64(nx, ny, nz, dv, psf, lsf, mode, u, p, want_cube):
    """Maps [n][3][ny][nx] (and cubes) of parameter sets p [n][10]."""
    dev = p.device
    sx, sz = u * psf / FWHM, (u * lsf / FWHM / dv if mode == 0 else 0.0)
    R, Rz = math.ceil(4 * sx) if sx > 0 else 0, math.ceil(4 * sz) if sz > 0 else 0
    f64 = dict(dtype=torch.float64, device=dev)
    at = lambda m, r: (torch.arange(-r, u * m + r, **f64) + 0.5) / u - 0.5  # noqa: E731  data coordinates
    x, y = at(nx, R).reshape(1, 1, -1), at(ny, R).reshape(1, -1, 1)
    vz = ((at(nz, Rz) - 0.5 * (nz - 1)) * dv).reshape(1, -1, 1, 1)
    c = [p[:, k].reshape(-1, 1, 1) for k in range(10)]
    pa, inc = torch.deg2rad(c[2]), torch.deg2rad(c[3])
    xe = -(x - c[0]) * torch.sin(pa) + (y - c[1]) * torch.cos(pa)
    yd = (-(x - c[0]) * torch.cos(pa) - (y - c[1]) * torch.sin(pa)) / torch.cos(inc)
    r = torch.sqrt(xe * xe + yd * yd)
    vlos = c[4] + 2.0 / math.pi * c[5] * torch.atan(r / c[6]) / r * xe * torch.sin(inc)
    s = c[7] if mode == 0 else torch.sqrt(c[7] ** 2 + (lsf / FWHM) ** 2)
    a = c[8] * torch.exp(-r / c[9]) * dv / (s * math.sqrt(2.0 * math.pi))
    cube = a[:, None] * torch.exp(-0.5 * ((vz - vlos[:, None]) / s[:, None]) ** 2)
    n, ez, ey, ex = cube.shape
    bx, by, bz = _band(_taps(sx, R, dev), u * nx), _band(_taps(sx, R, dev), u * ny), _band(_taps(sz, Rz, dev), u * nz)
    cube = torch.matmul(bz, cube.reshape(n, ez, ey * ex)).reshape(n, u * nz, ey, ex)
    cube = torch.matmul(by, cube)
    cube = torch.matmul(cube, bx.T)
    if u > 1:
        cube = cube.reshape(n, nz, u, ny, u, nx, u).mean(dim=(2, 4, 6))
    v = ((torch.arange(nz, **f64) - 0.5 * (nz - 1)) * dv).reshape(1, -1, 1, 1)
    m0 = cube.sum(1)
    ok = m0 > 1e-20 * c[8]
    d = torch.where(ok, m0, torch.ones_like(m0))
    m1 = (cube * v).sum(1) / d
    m2 = torch.sqrt((cube * (v - m1[:, None]) ** 2).sum(1) / d)
    maps = torch.stack([torch.where(ok, m0, 0.0), torch.where(ok, m1, c[4].expand_as(m1)), torch.where(ok, m2, 0.0)], 1)
    return (maps, cube) if want_cube else maps


def _geometry64(case):
    return [case[k] for k in ("nx", "ny", "nz", "dv", "psf", "lsf", "mode", "up")]


def _chunk(case):
    u = case["up"]
    voxels = (u * case["nx"] + 20 * u) * (u * case["ny"] + 20 * u) * (u * case["nz"] + 12 * u)
    return max(1, int(1.5e8 / voxels))


def _seed_forward64(w, v, sig, mask):
    m = mask.double()
    h = torch.stack([v.double() / 200.0 * m, sig.double() / 100.0 * m, m, torch.zeros_like(m)], 1)
    at = 0
    for l, (c, k) in enumerate(zip(CNN_C, CNN_K)):
        blk = w[at:at + c * (k + 1)].reshape(c, k + 1)
        at += c * (k + 1)
        wl, b = blk[:, :k], blk[:, k]
        if l < 4:
            h = torch.relu(torch.nn.functional.conv2d(h, wl.reshape(c, 2, 2, -1).permute(0, 3, 1, 2), b, stride=2))
        else:
            if l == 4:  # 4 x 4 x 256 in bit-interleaved order of (y, x)
                n = h.shape[0]
                h = h.reshape(n, 256, 2, 2, 2, 2).permute(0, 2, 4, 3, 5, 1).reshape(n, 4096)
            h = h @ wl.T + b
            h = torch.relu(h) if l == 4 else h
    return h


def exact(case, seed):
    dev, kind = _device(), case["kind"]
    if kind in ("maps", "eval", "cubes"):
        p = torch.from_numpy(_disc_params(case, seed)).to(dev)
        k, g = _chunk(case), _geometry64(case)
        if kind != "cubes":
            return {"maps": torch.cat([_model64(*g, p[i:i + k], False) for i in range(0, len(p), k)])}
        both = [_model64(*g, p[i:i + k], True) for i in range(0, len(p), k)]
        return {"cubes": torch.cat([b[1] for b in both]), "maps": torch.cat([b[0] for b in both])}
    if kind == "survey":
        out = []
        for g, p in zip(*_survey(case["n"], seed)):
            q = torch.from_numpy(p).reshape(1, 10).to(dev)
            out.append(_model64(g.nx, g.ny, g.nz, g.dv, g.psf_fwhm, g.lsf_fwhm, 0, 1, q, False).reshape(-1))
        return {"maps": torch.cat(out)}
    if kind == "jacobian":
        p = torch.from_numpy(_disc_params(case, seed)).to(dev)
        wv, ws, mask = _weights(case, seed, dev)
        w = (torch.stack([wv, ws]) * mask).double()
        k, g, out = max(1, _chunk(case) // 2), _geometry64(case), []
        for i in range(0, len(p), k):
            q = p[i:i + k]
            cols = []
            for j in range(10):
                t = torch.zeros_like(q)
                t[:, j] = 1.0
                cols.append(torch.func.jvp(lambda a: _model64(*g, a, False)[:, 1:] * w, (q,), (t,))[1])
            out.append(torch.stack(cols, 1))
        return {"jac": torch.cat(out)}
    if kind == "fit":
        return None
    v, sig, mask, t, w, m, u = _seed_data(case["n"], seed, dev)
    w = w.double().requires_grad_(kind == "train")
    y = _seed_forward64(w, v, sig, mask)
    if kind == "forward":
        return {"out": y}
    loss = ((y[:, :10] - t.double()) ** 2).mean()
    (g,) = torch.autograd.grad(loss, w)
    m, u, step = 0.9 * m.double() + 0.1 * g, 0.999 * u.double() + 0.001 * g * g, 1001
    new = w.detach() - LR * (m / (1 - 0.9 ** step)) / (torch.sqrt(u / (1 - 0.999 ** step)) + 1e-8)
    return {"weights": new, "adam_m": m, "adam_v": u, "loss": loss.detach().reshape(1)}
