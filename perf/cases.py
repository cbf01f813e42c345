"""The work a user has this library do, as measurable cases.

Each case is one pass of a part of a reconstruction through the package's public entry points:
the rasterizer and the voxelizer forward and backward (`project`, `project_batch`, `voxelize`,
`volume_tv`), the losses (`image_loss`, `ssim3d`), the FDK start (`fdk`), the brick MLP's
gradient (`mlp_grad`) and one whole optimisation step (`recon_step`).  `listed()` holds fixed
sizes from the package's own configurations and tests, `draw(rng)` further sizes of the same
ranges.  `exact()` restates every path in 64-bit torch from the method's definitions.
"""
import ctypes
import math

import numpy as np
import torch

import paper_2604_01844_gb300 as gsct
from paper_2604_01844_gb300 import binding as B
from paper_2604_01844_gb300.mlp import K_IN, N_OUT, N_OUT_PAD, BrickMLP
from paper_2604_01844_gb300.recon import PhantomProblem, ReconConfig, Reconstruction, fdk_volume

DEV = "cuda"
D_SO, D_OD, DET = 4.0, 2.0, 3.0  # source and detector distances from the axis, detector side
ALPHA_SSIM, ALPHA_TV = 0.25, 0.05
FIT_ALPHA = 0.2


def listed():
    return [
        # the smallest useful call: 2,000 Gaussians, 8 views of 64^2; launches and latency count
        dict(name="project_tiny", kind="project", beam="cone", views=8, W=64, H=64, n=2000,
             scale=0.02, tile=16, eps=0.0),
        # the projection of the standard reconstruction step (75 views of 512^2)
        dict(name="project_512", kind="project", beam="cone", views=75, W=512, H=512, n=50000,
             scale=0.012, tile=16, eps=0.0),
        # the large detector, with the tile the autotuner picks there
        dict(name="project_1024", kind="project", beam="cone", views=75, W=1024, H=1024,
             n=200000, scale=0.008, tile=32, eps=0.0),
        # parallel beam, a detector that no tile divides, a density cut
        dict(name="project_parallel", kind="project", beam="parallel", views=41, W=389, H=517,
             n=30011, scale=0.015, tile=16, eps=1e-3),
        # sixteen small uneven reconstructions projected in one call
        dict(name="project_batch16", kind="project_batch", instances=16, views=32, det=192,
             n=6000, scale=0.02, tile=16),
        # the TV branch of every reconstruction step: voxelize, TV, voxelizer backward
        dict(name="volume_tv_256", kind="volume_tv", dims=256, n=50000, scale=0.012, brick=16),
        # the voxelizer of the volume fit at its full size
        dict(name="voxelize_1024", kind="voxelize", nx=1024, ny=1024, nz=1024, n=500000,
             scale=0.004, brick=16),
        # L1 + D-SSIM of the standard step's projections
        dict(name="image_loss_512", kind="image_loss", views=75, W=512, H=512),
        # the volume fit's SSIM loss and gradient
        dict(name="ssim3d_384", kind="ssim3d", nx=384, ny=384, nz=384),
        # the FDK volume every reconstruction starts from
        dict(name="fdk_256", kind="fdk", views=75, W=512, H=512, dims=256),
        # the gradient of a training batch of the brick MLP (forward, render loss, backward)
        dict(name="mlp_grad_1024", kind="mlp_grad", bricks=1024),
        # one whole optimisation step
        dict(name="recon_step_512", kind="recon_step", views=75, side=512, dims=256, n=50000,
             scale=0.012),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["project", "project", "project", "project_batch", "volume_tv", "voxelize",
                       "voxelize", "image_loss", "ssim3d", "fdk", "recon_step", "mlp_grad"])
    big = {c["kind"]: max(work(x)["flops"] for x in listed() if x["kind"] == c["kind"])
           for c in listed()}
    while True:
        if kind == "project":
            c = dict(kind=kind, beam=rng.choice(["cone", "cone", "parallel"]),
                     views=_log(rng, 1, 75), W=_log(rng, 64, 1024), H=0, n=_log(rng, 2000, 200000),
                     scale=round(rng.uniform(0.006, 0.025), 4), tile=rng.choice([8, 16, 16, 32]),
                     eps=rng.choice([0.0, 0.0, 1e-3]))
            c["H"] = max(48, int(c["W"] * rng.uniform(0.6, 1.4)))
            if c["H"] > 1100:
                continue
        elif kind == "project_batch":
            c = dict(kind=kind, instances=rng.randint(2, 32), views=_log(rng, 4, 48),
                     det=_log(rng, 64, 256), n=_log(rng, 1000, 10000),
                     scale=round(rng.uniform(0.012, 0.03), 4), tile=rng.choice([8, 16, 16, 32]))
        elif kind == "volume_tv":
            c = dict(kind=kind, dims=_log(rng, 32, 384), n=_log(rng, 2000, 100000),
                     scale=round(rng.uniform(0.006, 0.02), 4), brick=rng.choice([16, 16, 32]))
        elif kind == "voxelize":
            a = _log(rng, 48, 700)
            c = dict(kind=kind, nx=a, ny=max(32, int(a * rng.uniform(0.7, 1.3))),
                     nz=max(32, int(a * rng.uniform(0.5, 1.2))), n=_log(rng, 2000, 300000),
                     scale=round(rng.uniform(0.004, 0.02), 4), brick=rng.choice([16, 16, 32, 64]))
        elif kind == "image_loss":
            c = dict(kind=kind, views=_log(rng, 1, 75), W=_log(rng, 64, 700), H=0)
            c["H"] = max(48, int(c["W"] * rng.uniform(0.6, 1.4)))
            if rng.random() < 0.6:
                c["W"] = (c["W"] + 3) // 4 * 4
        elif kind == "ssim3d":
            a = _log(rng, 48, 384)
            c = dict(kind=kind, nx=a, ny=max(32, int(a * rng.uniform(0.7, 1.2))),
                     nz=max(16, int(a * rng.uniform(0.4, 1.2))))
            if rng.random() < 0.7:
                c["nx"] = (c["nx"] + 3) // 4 * 4
        elif kind == "fdk":
            c = dict(kind=kind, views=_log(rng, 8, 75), W=_log(rng, 96, 640), H=0,
                     dims=_log(rng, 48, 256))
            c["H"] = max(64, int(c["W"] * rng.uniform(0.7, 1.3)))
        elif kind == "recon_step":
            c = dict(kind=kind, views=_log(rng, 8, 75), side=_log(rng, 64, 512),
                     dims=_log(rng, 48, 256), n=_log(rng, 2000, 50000),
                     scale=round(rng.uniform(0.01, 0.02), 4))
        else:
            return dict(kind=kind, bricks=128 * rng.randint(1, 24))
        if work(c)["flops"] <= big[kind]:
            return c


# ------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _gaussians(g, n, scale, radius=0.8, sigma_log=0.4):
    """Centres uniform in a ball, log-normal scales, uniform rotations, densities U(0.05, 1)."""
    d = torch.randn(n, 3, generator=g, device=DEV)
    r = radius * torch.rand(n, 1, generator=g, device=DEV) ** (1 / 3)
    rho = 0.05 + 0.95 * torch.rand(n, 1, generator=g, device=DEV)
    mr = torch.cat([d / d.norm(dim=1, keepdim=True) * r, rho], 1).contiguous()
    sc = torch.zeros(n, 4, device=DEV)
    sc[:, :3] = scale * torch.exp(sigma_log * torch.randn(n, 3, generator=g, device=DEV))
    q = torch.randn(n, 4, generator=g, device=DEV)
    return mr, sc, (q / q.norm(dim=1, keepdim=True)).contiguous()


def _views(beam, nv, W, H):
    pitch = DET / max(W, H)
    out = np.zeros(nv, dtype=B.VIEW_DTYPE)
    for k in range(nv):
        th = (2 * np.pi if beam == "cone" else np.pi) * k / nv
        c, s = np.cos(th), np.sin(th)
        out[k]["src"] = (D_SO * c, D_SO * s, 0) if beam == "cone" else (-c, -s, 0)
        out[k]["det_center"] = (-D_OD * c, -D_OD * s, 0)
        out[k]["u"], out[k]["v"] = (-s * pitch, c * pitch, 0), (0, 0, pitch)
        out[k]["mode"] = B.GS_CONE if beam == "cone" else B.GS_PARALLEL
    return out


def _grid(nx, ny, nz):
    g = np.zeros((), dtype=B.GRID_DTYPE)
    h = 2.0 / max(nx, ny, nz)
    g["dims"], g["voxel"] = (nx, ny, nz), (h, h, h)
    g["origin"] = (-0.5 * h * nx, -0.5 * h * ny, -0.5 * h * nz)
    return g


def _batch_sizes(case):
    """(views, W, H, n) of each instance, between half and all of the case's largest."""
    out = []
    for k in range(case["instances"]):
        r = np.random.default_rng(k)
        nv, W, H, n = (int(r.integers((case[f] + 1) // 2, case[f] + 1))
                       for f in ("views", "det", "det", "n"))
        out.append((nv, W, H, n))
    return out


def _smooth(g, shape):
    """A smooth positive field with values in about [0, 1] and some noise (last axis fastest)."""
    low = torch.rand(1, 1, *[max(2, s // 16) for s in shape[-len(shape):]], generator=g, device=DEV)
    mode = "bilinear" if len(shape) == 2 else "trilinear"
    f = torch.nn.functional.interpolate(low, size=shape, mode=mode, align_corners=True)[0, 0]
    return f + 0.02 * torch.rand(shape, generator=g, device=DEV)


def _pair_fields(g, shape):
    """A target and an estimate of it that is a few per cent off."""
    y = _smooth(g, shape)
    x = y * (0.97 + 0.06 * _smooth(g, shape)) + 0.01 * torch.randn(shape, generator=g, device=DEV)
    return x.contiguous(), y.contiguous()


def _ellipsoids(seed, n=40):
    r = np.random.default_rng(seed)
    d = r.standard_normal((n, 3))
    c = d / np.linalg.norm(d, axis=1, keepdims=True) * 0.5 * r.random((n, 1)) ** (1 / 3)
    ax = r.uniform(0.05, 0.35, (n, 3))
    ax *= np.minimum(1, (0.85 - np.linalg.norm(c, axis=1)) / ax.max(1))[:, None]
    q = r.standard_normal((n, 4))
    return np.concatenate([c, ax, q / np.linalg.norm(q, axis=1, keepdims=True),
                           r.random((n, 1))], 1)


def _bricks(g, m):
    """Bricks of a volume with smooth interfaces, values in [0, 1] (inputs and targets)."""
    a = (torch.arange(16, device=DEV) + 0.5) / 8 - 1
    z, y, x = torch.meshgrid(a, a, a, indexing="ij")
    p = torch.stack([x, y, z]).reshape(3, -1)
    nrm = torch.nn.functional.normalize(torch.randn(m, 3, generator=g, device=DEV), dim=1)
    side = torch.sigmoid(6 * (nrm @ p - torch.randn(m, 1, generator=g, device=DEV) * 0.6))
    lo, hi = torch.rand(m, 1, generator=g, device=DEV), torch.rand(m, 1, generator=g, device=DEV)
    t = lo + (hi - lo) * side
    noise = 0.03 * torch.randn(m, K_IN, generator=g, device=DEV)
    return (t + noise).to(torch.bfloat16).contiguous(), t.contiguous()


def prepare(case, seed):
    g, kind = _gen(seed), case["kind"]
    s = dict(case=case)
    if kind == "project":
        s["p"] = _gaussians(g, case["n"], case["scale"])
        s["proj"] = gsct.Projector(_views(case["beam"], case["views"], case["W"], case["H"]),
                                   case["W"], case["H"], tile=case["tile"], eps=case["eps"])
        s["proj"].ensure_capacity(*s["p"])
        s["dimg"] = torch.randn(case["views"], case["H"], case["W"], generator=g, device=DEV)
    elif kind == "project_batch":
        sizes = _batch_sizes(case)
        ps = [_gaussians(g, n, case["scale"]) for _, _, _, n in sizes]
        s["counts"] = [n for _, _, _, n in sizes]
        s["p"] = tuple(torch.cat(t) for t in zip(*ps))
        s["proj"] = gsct.BatchProjector([(_views("cone", nv, W, H), W, H)
                                         for nv, W, H, _ in sizes], tile=case["tile"])
        s["proj"].ensure_capacity(*s["p"], s["counts"])
        s["dimg"] = torch.randn(s["proj"].img_numel, generator=g, device=DEV)
    elif kind in ("volume_tv", "voxelize"):
        nx, ny, nz = _dims(case)
        s["p"] = _gaussians(g, case["n"], case["scale"])
        s["vox"] = gsct.Voxelizer(_grid(nx, ny, nz), brick=case["brick"])
        s["vox"].ensure_capacity(*s["p"])
        if kind == "voxelize":
            s["dvol"] = torch.randn(nz, ny, nx, generator=g, device=DEV)
        else:
            s["dvol"] = torch.empty(nz, ny, nx, device=DEV)
            s["loss"] = torch.zeros(1, device=DEV)
    elif kind == "image_loss":
        fields = [_pair_fields(g, (case["H"], case["W"])) for _ in range(min(4, case["views"]))]
        pick = [k % len(fields) for k in range(case["views"])]
        noise = 0.005 * torch.randn(case["views"], case["H"], case["W"], generator=g, device=DEV)
        s["x"] = torch.stack([fields[k][0] for k in pick]) + noise
        s["y"] = torch.stack([fields[k][1] for k in pick])
        s["range"] = float(s["y"].max())
        s["grad"] = torch.empty_like(s["x"])
        s["loss"] = torch.zeros(1, device=DEV)
        s["ws"] = torch.empty(B.lib().gs_ssim_workspace_size(s["x"].numel()), dtype=torch.uint8,
                              device=DEV)
    elif kind == "ssim3d":
        s["x"], s["y"] = _pair_fields(g, (case["nz"], case["ny"], case["nx"]))
        s["range"] = float(s["y"].max())
        s["grad"] = torch.empty_like(s["x"])
        s["loss"] = torch.zeros(1, device=DEV)
        s["ws"] = torch.empty(B.lib().gs_ssim3d_workspace_size(s["x"].numel()),
                              dtype=torch.uint8, device=DEV)
    elif kind == "fdk":
        s["grid"] = _grid(case["dims"], case["dims"], case["dims"])
        s["scan"] = PhantomProblem(_ellipsoids(seed), _views("cone", case["views"], case["W"],
                                                             case["H"]), case["W"], case["H"],
                                   _grid(8, 8, 8))
    elif kind == "mlp_grad":
        s["mlp"] = BrickMLP(seed=int(seed) % 1000)
        s["x16"], s["target"] = _bricks(g, case["bricks"])
        s["dy"] = torch.zeros(case["bricks"], N_OUT_PAD, device=DEV)
        s["loss"] = torch.zeros(1, device=DEV)
    else:  # recon_step
        side = case["side"]
        views = _views("cone", case["views"], side, side)
        s["p"] = _gaussians(g, case["n"], case["scale"])
        s["q"] = _gaussians(g, case["n"], case["scale"])
        target = gsct.Projector(views, side, side).forward(*s["q"])
        # the learning rates at the end of a decayed schedule
        cfg = ReconConfig(alpha_ssim=ALPHA_SSIM, alpha_tv=ALPHA_TV, lr_mean=2e-6, lr_rho=1e-4,
                          lr_scale=5e-5, lr_quat=1e-5)
        s["cfg"], s["range"] = cfg, float(target.max())
        s["rec"] = Reconstruction(views, side, side, target, _grid(*3 * (case["dims"],)),
                                  *[t.cpu().numpy() for t in s["p"]], cfg=cfg,
                                  data_range=s["range"])
    return s


def _dims(case):
    return 3 * (case["dims"],) if "dims" in case else (case["nx"], case["ny"], case["nz"])


# ------------------------------------------------------------------------------------------
# one pass
# ------------------------------------------------------------------------------------------
def run(s):
    case, kind = s["case"], s["case"]["kind"]
    L, st = B.lib(), B.stream_handle()
    if kind == "project":
        img = s["proj"].forward(*s["p"])
        return dict(img=img, grads=s["proj"].backward(*s["p"], s["dimg"]))
    if kind == "project_batch":
        img = s["proj"].forward(*s["p"], s["counts"])
        grads = s["proj"].backward(*s["p"], s["counts"], s["dimg"])
        return dict(img=s["proj"].split(img), grads=grads)
    if kind == "voxelize":
        vol = s["vox"].forward(*s["p"])
        return dict(vol=vol, grads=s["vox"].backward(*s["p"], s["dvol"]))
    if kind == "volume_tv":
        vol = s["vox"].forward(*s["p"])
        nz, ny, nx = vol.shape
        B.check(L.gs_memset(B.ptr(s["loss"]), 0, 4, st), "gs_memset")
        B.check(L.gs_tv3d_loss(B.ptr(vol), nx, ny, nz, ALPHA_TV, B.ptr(s["loss"]),
                               B.ptr(s["dvol"]), 0, st), "gs_tv3d_loss")
        grads = s["vox"].backward(*s["p"], s["dvol"])
        return dict(vol=vol, loss=s["loss"], dvol=s["dvol"], grads=grads)
    if kind in ("image_loss", "ssim3d"):
        x, y, ws = s["x"], s["y"], s["ws"]
        B.check(L.gs_memset(B.ptr(s["loss"]), 0, 4, st), "gs_memset")
        if kind == "image_loss":
            nv, H, W = x.shape
            B.check(L.gs_l1_ssim2d_loss(B.ptr(x), B.ptr(y), nv, H, W, s["range"], 1.0,
                                        ALPHA_SSIM, B.ptr(s["loss"]), B.ptr(s["grad"]), 0,
                                        B.ptr(ws), ws.numel(), st), "gs_l1_ssim2d_loss")
        else:
            nz, ny, nx = x.shape
            B.check(L.gs_ssim3d_loss(B.ptr(x), B.ptr(y), nx, ny, nz, s["range"], FIT_ALPHA,
                                     B.ptr(s["loss"]), B.ptr(s["grad"]), 0, B.ptr(ws),
                                     ws.numel(), st), "gs_ssim3d_loss")
        return dict(loss=s["loss"], grad=s["grad"])
    if kind == "fdk":
        return fdk_volume(s["scan"], s["grid"])
    if kind == "mlp_grad":
        mlp, m = s["mlp"], case["bricks"]
        y = mlp.forward(s["x16"])
        B.check(L.gs_memset(B.ptr(s["loss"]), 0, 4, st), "gs_memset")
        B.check(L.gs_brick_loss(B.ptr(y), N_OUT_PAD, B.ptr(s["target"]), m, B.ptr(s["loss"]),
                                B.ptr(s["dy"]), N_OUT_PAD, None, st), "gs_brick_loss")
        mlp.backward(s["dy"])
        return dict(y=y, loss=s["loss"], dy=s["dy"], grads=mlp.flat_grad)
    rec = s["rec"]
    loss = rec.step()
    return dict(loss=loss, img=rec.img, vol=rec.vol, grads=list(rec.grads), raw=list(rec.raw))


# ------------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------------
EVAL_FLOPS = 7 + 20  # FP32 operations of one in-cut evaluation, forward and backward


def _pixel_evals(views, W, H, n, scale, mag=(D_SO + D_OD) / D_SO):
    """In-cut (pixel, Gaussian) pairs of random Gaussians: the 3-sigma ellipses' areas."""
    r = scale * mag * max(W, H) / DET
    return views * n * 9 * math.pi * r * r * 1.24


def _voxel_evals(dims, n, scale):
    r = scale * max(dims) / 2
    return n * 36 * math.pi * r ** 3 * 1.27


def work(case):
    kind = case["kind"]
    if kind == "project":
        px = case["views"] * case["W"] * case["H"]
        mag = (D_SO + D_OD) / D_SO if case["beam"] == "cone" else 1.0
        ev = _pixel_evals(case["views"], case["W"], case["H"], case["n"], case["scale"], mag)
        return dict(bytes=8 * px + 96 * case["n"], flops=EVAL_FLOPS * ev)
    if kind == "project_batch":
        sizes = _batch_sizes(case)
        px, n = sum(v * W * H for v, W, H, _ in sizes), sum(x[3] for x in sizes)
        ev = sum(_pixel_evals(*x, case["scale"]) for x in sizes)
        return dict(bytes=8 * px + 96 * n, flops=EVAL_FLOPS * ev)
    if kind in ("voxelize", "volume_tv"):
        d = _dims(case)
        nv = d[0] * d[1] * d[2]
        ev = _voxel_evals(d, case["n"], case["scale"])
        return dict(bytes=8 * nv + 96 * case["n"],
                    flops=EVAL_FLOPS * ev + (12 * nv if kind == "volume_tv" else 0))
    if kind == "image_loss":
        px = case["views"] * case["W"] * case["H"]
        return dict(bytes=12 * px, flops=370 * px)
    if kind == "ssim3d":
        nv = case["nx"] * case["ny"] * case["nz"]
        return dict(bytes=12 * nv, flops=520 * nv)
    if kind == "fdk":
        px, nv = case["views"] * case["W"] * case["H"], case["dims"] ** 3
        return dict(bytes=4 * (px + nv),
                    flops=30 * nv * case["views"] + 10 * px * math.log2(2 * case["W"]))
    if kind == "mlp_grad":
        m = case["bricks"]
        layers = [(K_IN, 256), (256, 256), (256, 256), (256, N_OUT_PAD)]
        weights = sum(a * b for a, b in layers)
        fl = 2 * m * (2 * weights + weights - K_IN * 256) + EVAL_FLOPS * m * 12500
        return dict(bytes=m * (2 * K_IN + 4 * K_IN + 8 * N_OUT_PAD) + 6 * weights, flops=fl)
    px, nv = case["views"] * case["side"] ** 2, case["dims"] ** 3
    ev = _pixel_evals(case["views"], case["side"], case["side"], case["n"], case["scale"])
    ev += _voxel_evals(3 * (case["dims"],), case["n"], case["scale"])
    return dict(bytes=8 * px + 4 * nv + 400 * case["n"],
                flops=EVAL_FLOPS * ev + 370 * px + 12 * nv)


# ------------------------------------------------------------------------------------------
# the same in 64 bits, from the method's definitions
# ------------------------------------------------------------------------------------------
def _rot64(q):
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    r = [1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
         2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
         2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]
    return torch.stack(r, 1).view(-1, 3, 3)


def _footprint64(mr, sc, q, view, W, H):
    """(px, py, A, conic a, b, c, covariance xx, yy) of every Gaussian in one view."""
    t = lambda f: torch.tensor(np.asarray(view[f], dtype=np.float64), device=DEV)  # noqa: E731
    u, v, det, src = t("u"), t("v"), t("det_center"), t("src")
    pu, pv = u.norm(), v.norm()
    eu, ev = u / pu, v / pv
    cone = int(view["mode"]) == B.GS_CONE
    o = src if cone else det
    n = (det - src) / (det - src).norm() if cone else torch.linalg.cross(eu, ev)
    M = torch.stack([eu, ev, n])
    xc = (mr[:, :3] - o) @ M.T
    R = _rot64(q)
    if cone:
        D, (x, y, z) = (det - src).norm(), xc.unbind(1)
        one = torch.zeros_like(z)
        T = torch.stack([torch.stack([D / z, one, -D * x / z ** 2], 1),
                         torch.stack([one, D / z, -D * y / z ** 2], 1)], 1) @ M
        uu, vv, det_j = D * x / z, D * y / z, D * D * xc.norm(dim=1) / z ** 3
    else:
        T = M[:2].expand(len(mr), 2, 3)
        uu, vv, det_j = xc[:, 0], xc[:, 1], torch.ones_like(xc[:, 0])
    K = (T @ R) * sc[:, None, :3]
    S = K @ K.transpose(1, 2)
    det2 = S[:, 0, 0] * S[:, 1, 1] - S[:, 0, 1] ** 2
    A = mr[:, 3] * math.sqrt(2 * math.pi) * det_j * sc[:, :3].prod(1) / det2.sqrt()
    xx, xy, yy = S[:, 0, 0] / pu ** 2, S[:, 0, 1] / (pu * pv), S[:, 1, 1] / pv ** 2
    d = xx * yy - xy * xy
    return uu / pu + W / 2 - 0.5, vv / pv + H / 2 - 0.5, A, yy / d, -xy / d, xx / d, xx, yy


def _chunks(side, dim):
    """Index sets of Gaussians whose box side rounds up to the same size, a bounded number of
    box cells at a time."""
    k = ((side + 7) // 8 * 8).clamp(min=8)
    for s in torch.unique(k).tolist():
        ids = torch.nonzero(k == s)[:, 0]
        step = max(1, int(2 ** 26 / s ** dim))
        for a in range(0, len(ids), step):
            yield int(s), ids[a:a + step]


def _project64(p, views, W, H, eps, dimg=None, img=None):
    """Images, and the gradient of sum(img dimg) if dimg is given (a callable of the view)."""
    p = [t.double().requires_grad_() for t in p]
    out = torch.zeros(len(views), H * W, dtype=torch.float64, device=DEV)
    grads = [torch.zeros_like(t) for t in p]
    for k, view in enumerate(views):
        f = _footprint64(*p, view, W, H)
        px, py, A, a, b, c, xx, yy = [t.detach() for t in f]
        Q = torch.full_like(A, 9.0)
        if eps > 0:
            Q = torch.minimum(Q, 2 * torch.log((A.abs() / eps).clamp(min=1e-300)))
        live = Q > 0
        rx, ry = (Q.clamp(min=0) * xx).sqrt(), (Q.clamp(min=0) * yy).sqrt()
        live &= (px + rx >= 0) & (px - rx <= W - 1) & (py + ry >= 0) & (py - ry <= H - 1)
        side = (2 * torch.maximum(rx, ry)).ceil().long() + 2
        mom = torch.zeros(6, len(A), dtype=torch.float64, device=DEV)
        for s, ids in _chunks(torch.where(live, side, torch.zeros_like(side)), 2):
            ids = ids[live[ids]]
            if not len(ids):
                continue
            j = torch.arange(s, device=DEV)
            x0, y0 = (px[ids] - rx[ids]).floor().long(), (py[ids] - ry[ids]).floor().long()
            X, Y = x0[:, None, None] + j[None, None, :], y0[:, None, None] + j[None, :, None]
            dx, dy = X - px[ids, None, None], Y - py[ids, None, None]
            q = a[ids, None, None] * dx * dx + 2 * b[ids, None, None] * dx * dy + \
                c[ids, None, None] * dy * dy
            on = (q < Q[ids, None, None]) & (X >= 0) & (X < W) & (Y >= 0) & (Y < H)
            e = torch.where(on, torch.exp(-0.5 * q), torch.zeros_like(q))
            at = (Y.clamp(0, H - 1) * W + X.clamp(0, W - 1)).expand_as(e)
            out[k].index_add_(0, at.reshape(-1), (A[ids, None, None] * e).reshape(-1))
            if dimg is not None:
                ge = dimg(k).reshape(-1)[at] * e
                mom[:, ids] = torch.stack([m.sum((1, 2)) for m in (
                    ge, ge * dx, ge * dy, ge * dx * dx, ge * dx * dy, ge * dy * dy)])
        if dimg is not None:
            m0, mx, my, mxx, mxy, myy = mom
            gf = (A * (a * mx + b * my), A * (b * mx + c * my), m0, -0.5 * A * mxx, -A * mxy,
                  -0.5 * A * myy)
            for t, g in zip(grads, torch.autograd.grad(f[:6], p, gf)):
                t += g
    return out.view(len(views), H, W), grads


def _voxelize64(p, grid, dvol=None):
    """Volume, and the gradient of sum(vol dvol) if dvol is given."""
    p = [t.double().requires_grad_() for t in p]
    nx, ny, nz = (int(v) for v in grid["dims"])
    o = torch.tensor(np.asarray(grid["origin"], dtype=np.float64), device=DEV)
    h = torch.tensor(np.asarray(grid["voxel"], dtype=np.float64), device=DEV)
    R = _rot64(p[2])
    S = (R / p[1][:, None, :3] ** 2) @ R.transpose(1, 2)
    ctr, rho, Si = p[0][:, :3].detach(), p[0][:, 3].detach(), S.detach()
    r = 3 * ((R * p[1][:, None, :3]).detach() ** 2).sum(2).sqrt()
    lim = torch.tensor([nx, ny, nz], device=DEV)
    lo, hi = ((ctr - r - o) / h - 0.5).floor().long(), ((ctr + r - o) / h - 0.5).ceil().long()
    live = ((hi >= 0) & (lo < lim)).all(1)
    vol = torch.zeros(nz * ny * nx, dtype=torch.float64, device=DEV)
    mom = torch.zeros(10, len(rho), dtype=torch.float64, device=DEV)
    side = (hi - lo).amax(1) + 1
    for s, ids in _chunks(torch.where(live, side, torch.zeros_like(side)), 3):
        ids = ids[live[ids]]
        if not len(ids):
            continue
        j = torch.arange(s, device=DEV)
        X, Y, Z = (lo[ids, k].view(-1, 1, 1, 1) + j.view(*sh) for k, sh in
                   enumerate(((1, 1, 1, -1), (1, 1, -1, 1), (1, -1, 1, 1))))
        dx, dy, dz = (o[k] + (I + 0.5) * h[k] - ctr[ids, k].view(-1, 1, 1, 1)
                      for k, I in enumerate((X, Y, Z)))
        m = lambda i, k: Si[ids, i, k].view(-1, 1, 1, 1)  # noqa: E731
        q = dx * (m(0, 0) * dx + 2 * m(0, 1) * dy + 2 * m(0, 2) * dz) + \
            dy * (m(1, 1) * dy + 2 * m(1, 2) * dz) + m(2, 2) * dz * dz
        on = (q < 9) & (X >= 0) & (X < nx) & (Y >= 0) & (Y < ny) & (Z >= 0) & (Z < nz)
        e = torch.where(on, torch.exp(-0.5 * q), torch.zeros_like(q))
        at = (Z.clamp(0, nz - 1) * ny + Y.clamp(0, ny - 1)) * nx + X.clamp(0, nx - 1)
        vol.index_add_(0, at.reshape(-1), (rho[ids].view(-1, 1, 1, 1) * e).reshape(-1))
        if dvol is not None:
            ge = dvol.reshape(-1)[at] * e
            mom[:, ids] = torch.stack([t.sum((1, 2, 3)) for t in (
                ge, ge * dx, ge * dy, ge * dz, ge * dx * dx, ge * dx * dy, ge * dx * dz,
                ge * dy * dy, ge * dy * dz, ge * dz * dz)])
    vol = vol.view(nz, ny, nx)
    if dvol is None:
        return vol, None
    g_ctr = rho[:, None] * torch.einsum("nij,jn->ni", Si, mom[1:4])
    gS = -0.5 * rho[:, None, None] * mom[4:][[0, 1, 2, 1, 3, 4, 2, 4, 5]].T.reshape(-1, 3, 3)
    g_sc, g_q = torch.autograd.grad(S, p[1:], gS)
    return vol, [torch.cat([g_ctr, mom[0][:, None]], 1), g_sc, g_q]


def _filter64(t, axes):
    w = torch.exp(-(torch.arange(11, dtype=torch.float64) - 5) ** 2 / (2 * 1.5 ** 2))
    w = (w / w.sum()).tolist()
    for ax in axes:
        n = t.shape[ax]
        pad = [0, 0] * (t.dim() - 1 - ax) + [5, 5]
        e = torch.nn.functional.pad(t, pad)
        t = sum(w[k] * e.narrow(ax, k, n) for k in range(11))
    return t


def _ssim_loss64(x, y, L, axes):
    c1, c2 = (0.01 * L) ** 2, (0.03 * L) ** 2
    mx, my = _filter64(x, axes), _filter64(y, axes)
    sxx, syy = _filter64(x * x, axes) - mx * mx, _filter64(y * y, axes) - my * my
    sxy = _filter64(x * y, axes) - mx * my
    return 1 - ((2 * mx * my + c1) * (2 * sxy + c2) /
                ((mx * mx + my * my + c1) * (sxx + syy + c2)))


def _image_loss64(x, y, L):
    """Value and gradient of mean |x - y| + alpha (1 - SSIM), some images at a time."""
    total, grad = 0.0, torch.empty_like(x, dtype=torch.float64)
    for a in range(0, len(x), 16):
        u, v = x[a:a + 16].double().detach().requires_grad_(), y[a:a + 16].double()
        f = ((u - v).abs().sum() + ALPHA_SSIM * _ssim_loss64(u, v, L, (2, 1)).sum()) / x.numel()
        grad[a:a + 16], = torch.autograd.grad(f, u)
        total = total + f.detach()
    return total.reshape(1), grad


def _tv64(vol):
    v = vol.detach().requires_grad_()
    f = sum(v.diff(dim=k).abs().sum() for k in range(3)) * (ALPHA_TV / v.numel())
    return f.detach().reshape(1), torch.autograd.grad(f, v)[0]


def _fdk64(proj, views, dims, grid):
    nv, H, W = proj.shape
    vol = torch.zeros(dims, dims, dims, dtype=torch.float64, device=DEV)
    o, h = np.asarray(grid["origin"], np.float64), np.asarray(grid["voxel"], np.float64)
    ax = [torch.as_tensor(o[k] + (np.arange(dims) + 0.5) * h[k], device=DEV) for k in range(3)]
    X, Y, Z = ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]
    i = torch.arange(W, device=DEV)
    for k, view in enumerate(views):
        g = {f: np.asarray(view[f], dtype=np.float64) for f in ("src", "det_center", "u", "v")}
        pu, pv = np.linalg.norm(g["u"]), np.linalg.norm(g["v"])
        eu, ev = g["u"] / pu, g["v"] / pv
        d = g["det_center"] - g["src"]
        Dsd = np.linalg.norm(d)
        n = d / Dsd
        Dso = -float(g["src"] @ n)
        tau = pu * Dso / Dsd
        us = ((i + 0.5 - W / 2) * tau).double()
        vs = (torch.arange(H, device=DEV) + 0.5 - H / 2).double() * (pv * Dso / Dsd)
        p = proj[k].double() * Dso / torch.sqrt(Dso ** 2 + us[None, :] ** 2 + vs[:, None] ** 2)
        m = (i[:, None] - i[None, :]).abs().double()
        ramp = torch.where(m % 2 == 1, -1 / (math.pi * tau * m.clamp(min=1)) ** 2,
                           torch.zeros_like(m))
        ramp.fill_diagonal_(1 / (4 * tau * tau))
        q = torch.nn.functional.pad((p @ ramp) * tau, (1, 1, 1, 1))
        r = [X - g["src"][0], Y - g["src"][1], Z - g["src"][2]]
        dot = lambda e: r[0] * e[0] + r[1] * e[1] + r[2] * e[2]  # noqa: E731
        U = dot(n)
        cx = Dsd * dot(eu) / U / pu + W / 2 - 0.5
        cy = Dsd * dot(ev) / U / pv + H / 2 - 0.5
        fx, fy = cx.floor(), cy.floor()
        wx, wy = cx - fx, cy - fy
        s = torch.zeros_like(cx)
        for a in (0, 1):
            for b in (0, 1):
                xi, yi = fx.long() + a + 1, fy.long() + b + 1  # in the padded image
                on = (xi >= 1) & (xi <= W) & (yi >= 1) & (yi <= H)
                val = q[yi.clamp(0, H + 1), xi.clamp(0, W + 1)]
                s += torch.where(on, val, torch.zeros_like(val)) * \
                    (wx if a else 1 - wx) * (wy if b else 1 - wy)
        vol += Dso ** 2 / U ** 2 * s
    return vol * (math.pi / nv)


def _brick_loss64(y, target):
    """Mean |render - target| over the bricks with their margin of 4 voxels."""
    m, r = len(y), y[:, :N_OUT].reshape(len(y), 32, 11)
    g = torch.arange(32, device=DEV)
    base = torch.stack([(g % 4 + 0.5) * 4, (g // 4 % 4 + 0.5) * 4, (g // 16 + 0.5) * 8], 1)
    half = torch.tensor([2.0, 2.0, 4.0], dtype=torch.float64, device=DEV)
    s0 = torch.tensor([1.2, 1.2, 2.4], dtype=torch.float64, device=DEV)
    c = base + half * torch.tanh(r[..., :3])
    sc = s0 * torch.exp(r[..., 3:6].clamp(-3, 2))
    q = r[..., 6:10] + torch.tensor([1.0, 0, 0, 0], dtype=torch.float64, device=DEV)
    R = _rot64(q.reshape(-1, 4)).view(m, 32, 3, 3)
    rho = torch.nn.functional.softplus(r[..., 10])
    a = torch.arange(24, device=DEV, dtype=torch.float64) - 3.5
    z, yy, x = torch.meshgrid(a, a, a, indexing="ij")
    pos = torch.stack([x, yy, z], -1).view(-1, 3)
    t = torch.zeros(m, 24, 24, 24, dtype=torch.float64, device=DEV)
    t[:, 4:20, 4:20, 4:20] = target.view(m, 16, 16, 16)
    v = 0
    for j in range(32):
        d = (pos[None] - c[:, j, None]) @ R[:, j] / sc[:, j, None]
        qq = (d * d).sum(-1)
        v = v + torch.where(qq < 9, rho[:, j, None] * torch.exp(-0.5 * qq), torch.zeros_like(qq))
    return (v - t.view(m, -1)).abs().sum()


def _mlp64(s):
    mlp, m = s["mlp"], s["case"]["bricks"]
    W = [w.double().requires_grad_() for w in mlp.W16]
    b = [t.double().requires_grad_() for t in mlp.b]
    h = s["x16"].double()
    for k in range(4):
        h = h @ W[k].T + b[k]
        h = torch.relu(h) if k < 3 else h
    y = h.detach().requires_grad_()
    dy, loss = torch.zeros_like(y), 0.0
    for a in range(0, m, 128):
        part = y.detach()[a:a + 128].requires_grad_()
        f = _brick_loss64(part, s["target"][a:a + 128].double()) / (m * 24 ** 3)
        dy[a:a + 128], = torch.autograd.grad(f, part)
        loss = loss + f.detach()
    g = torch.autograd.grad(h, W + b, dy)
    return dict(y=y.detach(), loss=loss.reshape(1), dy=dy, grads=torch.cat([t.flatten() for t in g]))


def _recon64(s):
    case, cfg = s["case"], s["cfg"]
    side, grid = case["side"], _grid(*3 * (case["dims"],))
    views = _views("cone", case["views"], side, side)
    img, _ = _project64(s["p"], views, side, side, 0.0)
    target, _ = _project64(s["q"], views, side, side, 0.0)
    loss, dimg = _image_loss64(img, target, s["range"])
    _, g1 = _project64(s["p"], views, side, side, 0.0, dimg=lambda k: dimg[k])
    vol, _ = _voxelize64(s["p"], grid)
    tv, dvol = _tv64(vol)
    _, g2 = _voxelize64(s["p"], grid, dvol)
    grads = [a + b for a, b in zip(g1, g2)]
    # the first Adam step on the raw parameters: softplus density, log scales
    p = [t.double() for t in s["p"]]
    raw = [p[0].clone(), torch.zeros_like(p[1]), p[2]]
    raw[0][:, 3] = torch.log(torch.expm1(p[0][:, 3]))
    raw[1][:, :3] = torch.log(p[1][:, :3])
    step = [g.clone() for g in grads]
    step[0][:, 3] *= torch.sigmoid(raw[0][:, 3])
    step[1][:, :3] *= p[1][:, :3]
    lr = [torch.tensor([cfg.lr_mean] * 3 + [cfg.lr_rho], device=DEV), cfg.lr_scale, cfg.lr_quat]
    raw = [r - k * g / (g.abs() + cfg.eps) for r, k, g in zip(raw, lr, step)]
    return dict(loss=loss + tv, img=img, vol=vol, grads=grads, raw=raw)


def exact(case, seed):
    kind = case["kind"]
    s = prepare(case, seed)
    if kind == "project":
        views = _views(case["beam"], case["views"], case["W"], case["H"])
        img, g = _project64(s["p"], views, case["W"], case["H"], case["eps"],
                            dimg=lambda k: s["dimg"][k].double())
        return dict(img=img, grads=tuple(g))
    if kind == "project_batch":
        imgs, grads, at = [], [], 0
        for (nv, W, H, n), d in zip(_batch_sizes(case), s["proj"].split(s["dimg"])):
            img, g = _project64([t[at:at + n] for t in s["p"]], _views("cone", nv, W, H), W, H,
                                0.0, dimg=lambda k: d[k].double())
            imgs.append(img)
            grads.append(g)
            at += n
        return dict(img=imgs, grads=tuple(torch.cat(t) for t in zip(*grads)))
    if kind == "voxelize":
        vol, g = _voxelize64(s["p"], _grid(*_dims(case)), s["dvol"].double())
        return dict(vol=vol, grads=tuple(g))
    if kind == "volume_tv":
        grid = _grid(*_dims(case))
        vol, _ = _voxelize64(s["p"], grid)
        loss, dvol = _tv64(vol)
        return dict(vol=vol, loss=loss, dvol=dvol, grads=tuple(_voxelize64(s["p"], grid, dvol)[1]))
    if kind == "image_loss":
        loss, grad = _image_loss64(s["x"], s["y"], s["range"])
        return dict(loss=loss, grad=grad)
    if kind == "ssim3d":
        x = s["x"].double().requires_grad_()
        f = FIT_ALPHA * _ssim_loss64(x, s["y"].double(), s["range"], (2, 1, 0)).mean()
        return dict(loss=f.detach().reshape(1), grad=torch.autograd.grad(f, x)[0])
    if kind == "fdk":
        return _fdk64(s["scan"].proj, _views("cone", case["views"], case["W"], case["H"]),
                      case["dims"], s["grid"])
    return _mlp64(s) if kind == "mlp_grad" else _recon64(s)
