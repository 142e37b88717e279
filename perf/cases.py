"""The work a user has this rasterizer do, as measurable cases.

`listed()` names the cases, `draw()` gives further ones of the same ranges, `prepare()` makes a
case's inputs on the GPU from a seed, `run()` is one pass through the public entry points, `work()`
counts what a pass cannot do without and `exact()` gives the same outputs in 64 bits, in plain torch
and without this package.

Scenes follow the repository's generators: a mixture of 64 anisotropic clusters seen from distance
4 (view synthesis; at fewer than a million Gaussians their size grows with n^(-1/3) and their density
falls by as much, so that they cover the scene as well), means uniform in a cube (the smallest
workload) and means uniform in the unit ball (tomography, voxel grids).
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2412_03378_gb300 as vg

DEV = "cuda"
SQRT_2PI = math.sqrt(2.0 * math.pi)
TAU_CUT = 1e-6


def listed():
    return [
        # one small frame, no gradient (a preview, a unit of a service): launches and latency count
        dict(name="frame_tiny", kind="frame", scene="uniform", n=2000, deg=0, storage="f32", mode="exact",
             width=128, height=128, views=1),
        # the paper's own parameters (Eq. 20 density, softplus colour) early in a training run, through
        # autograd, on an image whose size is no multiple of a tile
        dict(name="train_small", kind="train", scene="cluster", n=10007, deg=1, storage="f32", mode="theta",
             width=317, height=211, views=1),
        # an ordinary training step through autograd
        dict(name="train_100k", kind="train", scene="cluster", n=100000, deg=3, storage="f32", mode="compat",
             width=640, height=416, views=1),
        # the headline: a training loop on the library's calls, the loss fused into the forward, the
        # instance capacity reserved once
        dict(name="train_1m", kind="train_ws", scene="cluster", n=1000000, deg=3, storage="f32", mode="compat",
             width=1280, height=832, views=1),
        # serving a trained scene in 16-bit storage (FP32 means) at full HD
        dict(name="frame_hd_mixed", kind="frame", scene="cluster", n=1500000, deg=3, storage="mixed", mode="compat",
             width=1920, height=1080, views=1),
        # a batch of views of uneven size, 16-bit storage, forward and backward
        dict(name="train_views_mixed", kind="train_ws", scene="cluster", n=300000, deg=3, storage="mixed",
             mode="compat", width=901, height=603, views=4),
        # the 3DGS comparison mode, forward and backward
        dict(name="train_splat", kind="train", scene="cluster", n=50000, deg=2, storage="f32", mode="splat",
             width=500, height=333, views=1),
        # sparse-view tomography: few angles, a ragged detector, through autograd
        dict(name="tomo_sparse", kind="tomo", n=8000, angles=25, width=200, height=170),
        # a full-size tomography training step (several angle batches) with the loss fused
        dict(name="tomo_step", kind="tomo_step", n=200000, angles=64, width=512, height=512),
        # cone-beam projection and its gradient
        dict(name="cone_step", kind="cone", n=20000, views=12, width=256, height=256),
        # the density of a reconstruction on a regular grid
        dict(name="voxel_grid", kind="voxel", n=200000, nx=256, ny=256, nz=256),
        # the overlap-error map of a view: the blend against the ray-marched reference
        dict(name="march_map", kind="march", scene="uniform", n=2000, deg=0, storage="f32", mode="exact",
             width=320, height=208, views=1, samples=256),
    ]


def draw(rng):
    def span(lo, hi):   # whole numbers, spread over their logarithm
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("frame", "frame", "train", "train", "train_ws", "train_ws", "tomo", "tomo_step", "cone", "voxel",
                       "march"))
    if kind == "tomo":
        return dict(kind=kind, n=span(1000, 10000), angles=rng.randint(8, 30), width=rng.randint(64, 224),
                    height=rng.randint(64, 224))
    if kind == "tomo_step":
        return dict(kind=kind, n=span(5000, 200000), angles=rng.randint(16, 64), width=rng.randint(128, 512),
                    height=rng.randint(128, 512))
    if kind == "cone":
        return dict(kind=kind, n=span(2000, 50000), views=rng.randint(4, 16), width=rng.randint(96, 320),
                    height=rng.randint(96, 320))
    if kind == "voxel":
        return dict(kind=kind, n=span(5000, 200000), nx=rng.randint(48, 256), ny=rng.randint(48, 256),
                    nz=rng.randint(48, 256))
    if kind == "march":
        return dict(kind=kind, scene="uniform", n=span(500, 3000), deg=0, storage="f32", mode="exact",
                    width=rng.randint(96, 384), height=rng.randint(96, 256), views=1, samples=rng.randint(64, 320))
    view = dict(width=span(96, 1920), height=span(96, 1080))
    if kind == "frame":
        if rng.random() < 0.3:
            return dict(kind=kind, scene="uniform", n=span(500, 3000), deg=0, storage="f32", mode="exact",
                        width=rng.randint(64, 256), height=rng.randint(64, 256), views=1)
        return dict(kind=kind, scene="cluster", n=span(5000, 1500000), deg=rng.randint(1, 3),
                    storage=rng.choice(("f32", "mixed")), mode=rng.choice(("compat", "compat", "theta")), views=1, **view)
    if kind == "train":
        return dict(kind=kind, scene="cluster", n=span(5000, 300000), deg=rng.randint(1, 3), storage="f32",
                    mode=rng.choice(("compat", "theta", "splat")), width=span(96, 800), height=span(96, 600), views=1)
    return dict(kind=kind, scene="cluster", n=span(50000, 1000000), deg=3, storage=rng.choice(("f32", "mixed")),
                mode="compat", views=rng.randint(1, 4), width=span(200, 1280), height=span(150, 832))


# ------------------------------------------------------------------------------------ inputs

def _rand(g, shape, lo=0.0, hi=1.0):
    return torch.rand(shape, generator=g, device=DEV) * (hi - lo) + lo


def _shapes(g, n, lo, hi, kap_lo, kap_hi, flatten):
    """Scales, unit quaternions and densities; a share `flatten` of the Gaussians is thinned 100:1 on one axis."""
    scale = torch.exp(_rand(g, (n, 3), lo, hi))
    thin = _rand(g, (n,)) < flatten
    axis = torch.randint(0, 3, (n,), generator=g, device=DEV)
    scale[thin, axis[thin]] /= 100.0
    quat = torch.nn.functional.normalize(torch.randn((n, 4), generator=g, device=DEV), dim=1)
    kappa = torch.exp(_rand(g, (n,), math.log(kap_lo), math.log(kap_hi)))
    return scale, quat, kappa


def _view_scene(case, g):
    n, deg = case["n"], case["deg"]
    if case["scene"] == "uniform":
        mu = _rand(g, (n, 3), -1.0, 1.0)
        scale, quat, kappa = _shapes(g, n, -4.0, -2.0, 0.5, 50.0, 0.0)
    else:
        centre, spread = _rand(g, (64, 3), -0.8, 0.8), _rand(g, (64, 3), 0.05, 0.25)
        frame = _rotation(torch.nn.functional.normalize(torch.randn((64, 4), generator=g, device=DEV), dim=1))
        at = torch.randint(0, 64, (n,), generator=g, device=DEV)
        z = torch.randn((n, 3), generator=g, device=DEV) * spread[at]
        mu = (centre[at] + (frame[at] * z[:, None, :]).sum(-1)).clamp(-1.0, 1.0)
        grow = max(0.0, math.log(1e6 / n) / 3.0)
        scale, quat, kappa = _shapes(g, n, -6.0 + grow, -4.0 + grow, 0.1 * math.exp(-grow), 100.0 * math.exp(-grow), 0.2)
    if deg == 0:
        sh = _rand(g, (n, 1, 3), -math.sqrt(math.pi), math.sqrt(math.pi))
    else:
        sh = 0.2 * torch.randn((n, (deg + 1) ** 2, 3), generator=g, device=DEV)
    if case["mode"] == "theta":        # Eq. 20's theta
        kappa = _rand(g, (n,), 0.01, 0.99)
    elif case["mode"] == "splat":      # peak opacities
        kappa = 1.0 - torch.exp(-kappa * SQRT_2PI * torch.exp(torch.log(scale).mean(1)))
    if case["storage"] == "mixed":
        scale, quat, kappa, sh = scale.bfloat16(), quat.bfloat16(), kappa.bfloat16(), sh.half()
    return [t.contiguous() for t in (mu, scale, quat, kappa, sh)]


def _ball_scene(n, g):
    v = torch.nn.functional.normalize(torch.randn((n, 3), generator=g, device=DEV), dim=1)
    mu = v * _rand(g, (n, 1)) ** (1.0 / 3.0)
    return [mu.contiguous(), *_shapes(g, n, -5.0, -3.0, 0.1, 10.0, 0.0)]


def _camera(eye, width, height, hfov, down=(0.0, 1.0, 0.0)):
    eye, down = np.asarray(eye, np.float64), np.asarray(down, np.float64)
    fwd = -eye / np.linalg.norm(eye)
    if abs(float(down @ fwd)) > 0.99:
        down = np.array([0.0, 0.0, -1.0])
    right = np.cross(down, fwd)
    right /= np.linalg.norm(right)
    R = np.stack([right, np.cross(fwd, right), fwd])
    f = float(np.float32(0.5 * width / math.tan(0.5 * hfov)))
    return SimpleNamespace(R=R.astype(np.float32), t=(-R @ eye).astype(np.float32), fx=f, fy=f, cx=0.5 * width,
                           cy=0.5 * height, width=width, height=height)


def _cameras(case):
    """One camera in front of the scene, or several on a Fibonacci sphere whose images shrink from view to view."""
    if case["kind"] == "cone":
        fov, k = 2.0 * math.atan(1.1 / 4.0), case["views"]
        at = [2.0 * math.pi * i / k for i in range(k)]
        return [_camera((4.0 * math.cos(a), 4.0 * math.sin(a), 0.0), case["width"], case["height"], fov, (0.0, 0.0, -1.0))
                for a in at]
    cams, k = [], case["views"]
    for i in range(k):
        y = 1.0 - 2.0 * (i + 0.5) / k
        r, phi = math.sqrt(max(0.0, 1.0 - y * y)), math.pi * (3.0 - math.sqrt(5.0)) * i
        eye = (0.0, 0.0, -4.0) if k == 1 else (4.0 * math.cos(phi) * r, 4.0 * y, 4.0 * math.sin(phi) * r)
        cams.append(_camera(eye, max(32, case["width"] * (6 - i) // 6), max(32, case["height"] * (6 - i) // 6),
                            math.radians(60.0)))
    return cams


def _beam(case):
    w, h = case["width"], case["height"]
    pu, pv = (float(np.float32(2.0 / d)) for d in (w, h))
    angles = (np.arange(case["angles"]) * math.pi / case["angles"]).astype(np.float32)
    return SimpleNamespace(angles=angles, det_w=w, det_h=h, pitch_u=pu, pitch_v=pv, u0=-1.0, v0=-1.0)


def _opts(mode, flags=0):
    if mode == "exact":
        return vg.Opts.exact(flags=flags)
    if mode == "theta":
        return vg.Opts.compat(softplus_beta=10.0, bg=(0.2, 0.3, 0.4), flags=flags | vg.FLAG_DENSITY_THETA)
    if mode == "splat":
        return vg.Opts.compat(tau_cut=1.0 / 255.0, splat_dilation=0.3, flags=flags | vg.FLAG_SPLAT)
    return vg.Opts.compat(flags=flags)


def _inputs(case, seed):
    """The numbers of a case, the same for prepare() and exact()."""
    g = torch.Generator(DEV).manual_seed(int(seed))
    s = SimpleNamespace(kind=case["kind"], case=dict(case))
    if case["kind"] in ("tomo", "tomo_step", "cone", "voxel"):
        s.params = _ball_scene(case["n"], g)
    else:
        s.params = _view_scene(case, g)
    if case["kind"] in ("tomo", "tomo_step"):
        s.beam = _beam(case)
        s.target = _rand(g, (case["angles"], case["height"], case["width"]))
    elif case["kind"] != "voxel":
        s.cams = _cameras(case)
        s.pixels = sum(c.width * c.height for c in s.cams)
        s.target = _rand(g, (s.pixels,) if case["kind"] == "cone" else (s.pixels, 3))
    if case["kind"] == "voxel":
        s.dims = (case["nx"], case["ny"], case["nz"])
        s.voxel = tuple(2.0 / d for d in s.dims)
    if "target" in vars(s):
        s.scale = 1.0 / s.target.numel()
    return s


def _grads(params):
    return [torch.zeros(p.shape, device=DEV) for p in params]


def prepare(case, seed):
    s = _inputs(case, seed)
    k = case["kind"]
    if k in ("train", "tomo"):
        s.params = [p.requires_grad_(True) for p in s.params]
    if k == "train":
        s.ras = vg.Rasterizer(_opts(case["mode"]))
    elif k == "tomo":
        s.pro = vg.Projector()
    else:
        s.ws = vg.Workspace()
        sh = s.params[4] if len(s.params) == 5 else None
        s.g = vg.Gaussians(*s.params[:4], sh, case.get("deg", 0))
    if k in ("frame", "march", "train_ws"):
        s.rgb, s.T = torch.empty((s.pixels, 3), device=DEV), torch.empty(s.pixels, device=DEV)
    if k in ("frame", "march"):
        s.opts = _opts(case["mode"])
    if k == "march":
        s.mrgb, s.mT, s.err = (torch.empty(d, device=DEV) for d in ((s.pixels, 3), s.pixels, s.pixels))
    if k == "train_ws":   # the training loop's buffers; the instance capacity is reserved from one binning
        s.loss, s.dl, s.grads = torch.empty(1, device=DEV), torch.empty((s.pixels, 3), device=DEV), _grads(s.params)
        s.ws.preprocess(s.g, s.cams, _opts(case["mode"]))
        s.ws.bin_sort()
        q = s.ws.query()
        s.ws.reserve(q["n_items"], int(1.1 * q["n_instances"]) + 4096, q["n_pixels"], q["n_tiles"])
        s.opts = _opts(case["mode"], vg.FLAG_FIXED_CAPACITY | vg.FLAG_GRAD_ZERO)
    if k in ("tomo_step", "cone"):
        s.opts = vg.Opts(tau_cut=TAU_CUT, flags=vg.FLAG_GRAD_ZERO)
        s.loss, s.proj, s.grads = torch.empty(1, device=DEV), torch.empty_like(s.target), _grads(s.params)
    if k == "voxel":
        s.opts = vg.Opts(tau_cut=TAU_CUT)
        s.out = torch.empty(s.dims[::-1], device=DEV)
    return s


# ------------------------------------------------------------------------------------ one pass

def run(s):
    k = s.kind
    if k == "frame":
        s.ws.preprocess(s.g, s.cams, s.opts)
        s.ws.bin_sort()
        s.ws.render_fwd(s.rgb, s.T)
        return [s.rgb, s.T]
    if k == "train":
        rgb, T = s.ras.render(*s.params, s.cams)
        loss = s.scale * ((rgb - s.target) ** 2).sum()
        return [rgb.detach(), T.detach(), *torch.autograd.grad(loss, s.params)]
    if k == "train_ws":
        s.ws.preprocess(s.g, s.cams, s.opts)
        s.ws.bin_sort()
        s.ws.render_fwd_l2(s.rgb, s.T, s.target, s.scale, s.loss, s.dl)
        s.ws.render_bwd(s.dl, None, *s.grads)
        return [s.rgb, s.T, s.loss, *s.grads]
    if k == "tomo":
        proj = s.pro.parallel(*s.params, s.beam)
        loss = s.scale * ((proj - s.target) ** 2).sum()
        return [proj.detach(), *torch.autograd.grad(loss, s.params)]
    if k == "tomo_step":
        s.ws.tomo_l2_step(s.g, s.beam, s.opts, s.target, s.scale, s.proj, s.loss, *s.grads)
        return [s.proj, s.loss, *s.grads]
    if k == "cone":   # projection and gradient of a linear functional (`target` holds dL/dproj)
        s.ws.project_cone(s.g, s.cams, s.opts, s.proj, s.target, *s.grads)
        return [s.proj, *s.grads]
    if k == "voxel":
        s.ws.query_density(s.g, (-1.0, -1.0, -1.0), s.voxel, s.dims, s.opts, s.out)
        return [s.out]
    s.ws.preprocess(s.g, s.cams, s.opts)
    s.ws.bin_sort()
    s.ws.render_fwd(s.rgb, s.T)
    s.ws.ray_march(2.0, 6.0, s.case["samples"], s.mrgb, s.mT, s.rgb, s.err)
    return [s.rgb, s.T, s.mrgb, s.mT, s.err]


# ------------------------------------------------------------------------------------ the least work

def _sample(lo, hi, kap_lo, kap_hi, n=4096):
    """Scales, densities and ray directions in the Gaussians' frames, for expected footprints."""
    rng = np.random.Generator(np.random.PCG64(7))
    s, kap = np.exp(rng.uniform(lo, hi, (n, 3))), np.exp(rng.uniform(math.log(kap_lo), math.log(kap_hi), n))
    d = rng.standard_normal((n, 3))
    return s, kap, d / np.linalg.norm(d, axis=1, keepdims=True)


def _line_area(s, kap, d):
    """Expected area, in world units, of the footprint a Gaussian's line integral exceeds TAU_CUT on."""
    dn = np.linalg.norm(d / s, axis=1)                       # |S^-1 d|
    k2 = np.maximum(0.0, 2.0 * np.log(kap * SQRT_2PI / dn / TAU_CUT))
    return float(np.mean(math.pi * k2 * s.prod(1) * dn))     # sqrt(det of the 2D marginal) = s0 s1 s2 |S^-1 d|


def work(case):
    """Inputs read once, outputs written once.  Operations: those of each Gaussian and, where the sum
    has no early end, of each (pixel, Gaussian) pair that counts (11 for a line integral, 24 more for
    its gradient); the blended pairs of an early-stopping blend depend on the scene and are left out."""
    k, n = case["kind"], case["n"]
    if k in ("tomo", "tomo_step"):
        px = case["angles"] * case["width"] * case["height"]
        area = _line_area(*_sample(-5.0, -3.0, 0.1, 10.0)) * case["width"] * case["height"] / 4.0
        return {"bytes": 4 * (11 * n + px) + 4 * px + 4 * 11 * n, "flops": n * case["angles"] * (400 + 35 * area)}
    if k == "cone":
        px = case["views"] * case["width"] * case["height"]
        area = _line_area(*_sample(-5.0, -3.0, 0.1, 10.0)) * (case["width"] / 2.2) ** 2
        return {"bytes": 4 * (11 * n + px) + 4 * px + 4 * 11 * n, "flops": n * case["views"] * (800 + 65 * area)}
    if k == "voxel":
        s, kap, _ = _sample(-5.0, -3.0, 0.1, 10.0)
        vol = np.mean(4.0 / 3.0 * math.pi * np.maximum(0.0, 2.0 * np.log(kap / TAU_CUT)) ** 1.5 * s.prod(1))
        vox = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": 4 * 11 * n + 4 * vox, "flops": n * (200 + 16 * float(vol) * vox / 8.0)}
    px = sum(c.width * c.height for c in _cameras(case))
    rec = 28 if case["storage"] == "mixed" else 44
    sh = (case["deg"] + 1) ** 2 * 3
    par = n * (rec + sh * (2 if case["storage"] == "mixed" else 4))
    if k == "march":
        s, kap, d = _sample(-4.0, -2.0, 0.5, 50.0)
        pairs = n * _line_area(s, kap, d) * (case["width"] / (2.0 * 4.0 * math.tan(math.radians(30.0)))) ** 2
        steps = case["samples"] / 4.0 * float(np.mean(10.0 / np.linalg.norm(d / s, axis=1)))   # within 5 deviations
        return {"bytes": par + 36 * px, "flops": n * 400 + pairs * (60 + 11 * steps)}
    if k == "frame":
        return {"bytes": par + 16 * px, "flops": 400 * n * case["views"]}
    return {"bytes": par + 4 * n * (11 + sh) + (12 + 16) * px, "flops": 1200 * n * case["views"]}


# ------------------------------------------------------------------------------------ 64 bits

def _rotation(q):
    w, x, y, z = torch.nn.functional.normalize(q, dim=1).unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).reshape(-1, 3, 3)


def _harmonics(d, deg):
    x, y, z = d.unbind(1)
    pi = math.pi
    Y = [torch.full_like(x, 0.5 / math.sqrt(pi))]
    if deg > 0:
        c = math.sqrt(3 / (4 * pi))
        Y += [-c * y, c * z, -c * x]
    if deg > 1:
        a, b = math.sqrt(15 / (4 * pi)), math.sqrt(5 / (16 * pi))
        Y += [a * x * y, -a * y * z, b * (2 * z * z - x * x - y * y), -a * x * z, 0.5 * a * (x * x - y * y)]
    if deg > 2:
        e, f, h = math.sqrt(35 / (32 * pi)), math.sqrt(105 / (4 * pi)), math.sqrt(21 / (32 * pi))
        m = math.sqrt(7 / (16 * pi))
        Y += [-e * y * (3 * x * x - y * y), f * x * y * z, -h * y * (4 * z * z - x * x - y * y),
              m * z * (2 * z * z - 3 * x * x - 3 * y * y), -h * x * (4 * z * z - x * x - y * y),
              0.5 * f * z * (x * x - y * y), -e * x * (x * x - 3 * y * y)]
    return torch.stack(Y, 1)


def _colour(p, cam, deg, mode):
    R, t = (torch.as_tensor(v, device=DEV).double() for v in (cam.R, cam.t))
    d = torch.nn.functional.normalize(p[0] + (R.T @ t), dim=1)
    c = (_harmonics(d, deg)[:, :, None] * p[4]).sum(1) + 0.5
    return torch.nn.functional.softplus(c, beta=10.0, threshold=1e9) if mode == "theta" else c.clamp(min=0.0)


def _rows(p, cam, mode, colour):
    """Per Gaussian, differentiable, what a pixel needs: volumetric M (9), M mu_c (3), ln kappa sqrt(2 pi);
    splat mean (2), inverse covariance (3), ln o.  Then the colour."""
    R, t = (torch.as_tensor(v, device=DEV).double() for v in (cam.R, cam.t))
    mu, s, q, kap = p[:4]
    m = mu @ R.T + t
    B = R @ _rotation(q)
    if mode == "splat":
        u, v, iz = m[:, 0] / m[:, 2], m[:, 1] / m[:, 2], 1.0 / m[:, 2]
        J = torch.stack([torch.stack([cam.fx * iz, 0 * iz, -cam.fx * u * iz], 1),
                         torch.stack([0 * iz, cam.fy * iz, -cam.fy * v * iz], 1)], 1)
        F = J @ (B * s[:, None, :])
        S = F @ F.transpose(1, 2) + 0.3 * torch.eye(2, device=DEV, dtype=torch.float64)
        Q = torch.linalg.inv(S)
        r = [cam.fx * u + cam.cx - 0.5, cam.fy * v + cam.cy - 0.5, Q[:, 0, 0], Q[:, 0, 1], Q[:, 1, 1], torch.log(kap)]
        return torch.cat([torch.stack(r, 1), colour], 1)
    if mode == "theta":
        kap = -torch.log1p(-0.99 * kap) * (1.0 / s).sum(1) / 3.0
    M = B.transpose(1, 2) / s[:, :, None]
    return torch.cat([M.reshape(-1, 9), (M @ m[:, :, None])[:, :, 0], torch.log(kap * SQRT_2PI)[:, None], colour], 1)


def _boxes(p, cam, mode, cut):
    """Depths and pixel boxes (x0, y0, x1, y1) outside of which no pixel reaches `cut`."""
    R, t = (torch.as_tensor(v, device=DEV).double() for v in (cam.R, cam.t))
    mu, s, q, kap = p[:4]
    m = mu @ R.T + t
    B = (R @ _rotation(q)) * s[:, None, :]
    S, z = B @ B.transpose(1, 2), m[:, 2]
    if mode == "theta":
        kap = -torch.log1p(-0.99 * kap) * (1.0 / s).sum(1) / 3.0
    top = kap if mode == "splat" else kap * SQRT_2PI * s.max(1).values
    k2 = 2.0 * torch.log(top / cut) + 1.4
    seen = (z > 0.2) & (top > cut)
    lo, hi = [], []
    for a, f, c in ((0, cam.fx, cam.cx), (1, cam.fy, cam.cy)):
        if mode == "splat":
            r = m[:, a] / z
            h = torch.sqrt(k2.clamp(min=0) * ((f / z) ** 2 * (S[:, a, a] - 2 * r * S[:, a, 2] + r * r * S[:, 2, 2]) + 0.3))
            x0, x1 = f * r + c - 0.5 - h, f * r + c - 0.5 + h
        else:
            A, b, e = z * z - k2 * S[:, 2, 2], m[:, a] * z - k2 * S[:, a, 2], m[:, a] ** 2 - k2 * S[:, a, a]
            h, near = torch.sqrt((b * b - A * e).clamp(min=0)), A <= 0
            x0 = torch.where(near, torch.full_like(A, -1e9), f * (b - h) / A + c - 0.5)
            x1 = torch.where(near, torch.full_like(A, 1e9), f * (b + h) / A + c - 0.5)
        lo.append(x0 - 0.1)
        hi.append(x1 + 0.1)
    return z, torch.stack(lo + hi, 1), seen


def _tiles(cam, size, box, z, seen):
    """Pixel coordinates, image positions and depth-ordered Gaussians of every tile."""
    order = torch.argsort(z, stable=True)
    for ty in range(0, cam.height, size):
        in_y = seen & (box[:, 1] <= min(ty + size, cam.height) - 1) & (box[:, 3] >= ty)
        for tx in range(0, cam.width, size):
            in_x = in_y & (box[:, 0] <= min(tx + size, cam.width) - 1) & (box[:, 2] >= tx)
            y, x = torch.meshgrid(torch.arange(ty, min(ty + size, cam.height), device=DEV),
                                  torch.arange(tx, min(tx + size, cam.width), device=DEV), indexing="ij")
            x, y = x.reshape(-1), y.reshape(-1)
            yield x, y, y * cam.width + x, order[in_x[order]]


def _ray(cam, x, y):
    return torch.stack([(x + 0.5 - cam.cx) / cam.fx, (y + 0.5 - cam.cy) / cam.fy, torch.ones_like(x, dtype=torch.float64)], 1)


def _tau(r, cam, x, y, mode):
    """Optical depths [n, pixels] of the Gaussians' rows."""
    if mode == "splat":
        dx, dy = x[None, :] - r[:, 0:1], y[None, :] - r[:, 1:2]
        a = torch.exp(r[:, 5:6] - 0.5 * (r[:, 2:3] * dx * dx + 2 * r[:, 3:4] * dx * dy + r[:, 4:5] * dy * dy))
        return -torch.log1p(-a.clamp(max=0.99))
    d = _ray(cam, x, y)
    dp = torch.einsum("nij,pj->npi", r[:, :9].reshape(-1, 3, 3), d)
    cr = torch.cross(r[:, None, 9:12].expand_as(dp), dp, dim=2)
    a = (dp * dp).sum(2)
    return torch.exp(r[:, 12:13] + 0.5 * torch.log((d * d).sum(1)[None, :] / a) - 0.5 * (cr * cr).sum(2) / a)


def _blend(r, cam, x, y, mode):
    """Colour and transmittance of the pixels from depth-ordered rows (Eq. 14)."""
    tau = _tau(r, cam, x, y, mode)
    if mode != "exact":
        if mode != "splat":
            tau = tau.clamp(max=math.log(100.0))
        tau = tau * (tau.detach() >= -math.log1p(-1.0 / 255.0))
        before = torch.cumsum(tau.detach(), 0) - tau.detach()
        tau = tau * (torch.exp(-before) >= 1e-4)
    end = torch.cumsum(tau, 0)
    w = torch.exp(tau - end) - torch.exp(-end)
    T = torch.exp(-tau.sum(0))
    rgb = torch.einsum("np,nc->pc", w, r[:, -3:])
    if mode == "theta":
        rgb = rgb + T[:, None] * torch.tensor([0.2, 0.3, 0.4], device=DEV, dtype=torch.float64)
    return rgb, T


def _exact_views(s, p, mode, cut, grad, cone=False):
    """Image and transmittance of every view and, with `grad`, the gradients of the case's loss."""
    rgbs, Ts, total, at = [], [], [torch.zeros_like(v) for v in p], 0
    for cam in s.cams:
        leaf = [v.detach().requires_grad_(grad) for v in p]
        colour = torch.zeros((len(p[0]), 3), device=DEV, dtype=torch.float64) if cone else \
            _colour(leaf, cam, s.case["deg"], mode)
        rows = _rows(leaf, cam, mode, colour)
        flat, drow = rows.detach(), torch.zeros_like(rows)
        z, box, seen = _boxes(p, cam, mode, cut)
        rgb = torch.zeros((cam.width * cam.height, 3), device=DEV, dtype=torch.float64)
        T = torch.ones(cam.width * cam.height, device=DEV, dtype=torch.float64)
        for x, y, pix, ids in _tiles(cam, 16, box, z, seen):
            r = flat[ids].requires_grad_(grad)
            c, t = _blend(r, cam, x, y, mode)
            rgb[pix], T[pix] = c.detach(), t.detach()
            if grad and len(ids):
                goal = s.target[at + pix].double()
                loss = (goal * t).sum() if cone else s.scale * ((c - goal) ** 2).sum()
                drow.index_add_(0, ids, torch.autograd.grad(loss, r)[0])
        if grad:
            drow[~seen] = 0.0
            back = torch.autograd.grad(rows, leaf, drow, allow_unused=True)
            total = [a if b is None else a + b.nan_to_num(0.0) for a, b in zip(total, back)]
        rgbs.append(rgb)
        Ts.append(T)
        at += cam.width * cam.height
    return torch.cat(rgbs), torch.cat(Ts), total


def _exact_march(s, p, rgb):
    cam, k = s.cams[0], s.case["samples"]
    delta = 4.0 / k
    rows = _rows(p, cam, "exact", _colour(p, cam, 0, "exact"))
    z, box, seen = _boxes(p, cam, "exact", TAU_CUT)
    out, Tout = torch.zeros_like(rgb), torch.ones(len(rgb), device=DEV, dtype=torch.float64)
    t = 2.0 + (torch.arange(k, device=DEV, dtype=torch.float64) + 0.5) * delta
    for x, y, pix, ids in _tiles(cam, 8, box, z, seen):
        r, d = rows[ids], _ray(cam, x, y)
        d = d / d.norm(dim=1, keepdim=True)
        dp = torch.einsum("nij,pj->npi", r[:, :9].reshape(-1, 3, 3), d)
        a, op = (dp * dp).sum(2), r[:, None, 9:12]
        gam = (dp * op).sum(2) / a
        cr = torch.cross(op.expand_as(dp), dp, dim=2)
        lp = r[:, 12:13] - math.log(SQRT_2PI) - 0.5 * (cr * cr).sum(2) / a
        v = torch.exp(lp[:, :, None] - 0.5 * a[:, :, None] * (t - gam[:, :, None]) ** 2)
        sig, col = v.sum(0), torch.einsum("npk,nc->pkc", v, r[:, -3:])
        depth = torch.cumsum(sig, 1) * delta
        w = torch.exp(sig * delta - depth) * -torch.expm1(-sig * delta) / sig.clamp(min=1e-300)
        out[pix], Tout[pix] = (w[:, :, None] * col).sum(1), torch.exp(-depth[:, -1])
    return out, Tout, (out - rgb).abs().max(1).values


def _exact_tomo(s, p):
    b = s.beam
    du = torch.as_tensor(b.u0, device=DEV) + (torch.arange(b.det_w, device=DEV).double() + 0.5) * b.pitch_u
    dv = torch.as_tensor(b.v0, device=DEV) + (torch.arange(b.det_h, device=DEV).double() + 0.5) * b.pitch_v
    proj, total = [], [torch.zeros_like(v) for v in p]

    def tau(part, ct, st):
        mu, sc, q, kap = part
        F = _rotation(q) * sc[:, None, :]
        eu, ev = (torch.tensor(e, device=DEV, dtype=torch.float64) for e in ((-st, ct, 0.0), (0.0, 0.0, 1.0)))
        fu, fv = (F * eu[:, None]).sum(1), (F * ev[:, None]).sum(1)
        c00, c01, c11 = (fu * fu).sum(1), (fu * fv).sum(1), (fv * fv).sum(1)
        det = torch.linalg.cross(fu, fv).square().sum(1)
        x, y = du[None, :] - (mu @ eu)[:, None], dv[None, :] - (mu @ ev)[:, None]
        A = torch.log(kap * SQRT_2PI * sc.prod(1)) - 0.5 * torch.log(det)
        e = A[:, None, None] - 0.5 * ((c00 / det)[:, None, None] * (y * y)[:, :, None] +
                                      (c11 / det)[:, None, None] * (x * x)[:, None, :])
        return torch.exp(e + (c01 / det)[:, None, None] * y[:, :, None] * x[:, None, :])

    for k, ang in enumerate(b.angles):
        ct, st = (float(np.float32(f(float(ang)))) for f in (math.cos, math.sin))
        parts = list(zip(*(v.split(1000) for v in p)))
        T = torch.exp(-sum(tau(part, ct, st).sum(0) for part in parts))
        proj.append(T)
        gtau = -2.0 * s.scale * (T - s.target[k].double()) * T
        for i, part in enumerate(parts):
            leaf = [v.detach().requires_grad_(True) for v in part]
            back = torch.autograd.grad((gtau * tau(leaf, ct, st).sum(0)).sum(), leaf)
            for a, g in zip(total, back):
                a[1000 * i:1000 * i + len(g)] += g
    return [torch.stack(proj), *total]


def _exact_voxel(s, p):
    mu, sc, q, kap = p
    R = _rotation(q)
    P = (R / (sc * sc)[:, None, :]) @ R.transpose(1, 2)
    half = torch.sqrt((2.0 * torch.log(kap / TAU_CUT) + 1.4).clamp(min=0)[:, None] *
                      ((R * sc[:, None, :]) ** 2).sum(2))
    h = [float(np.float32(v)) for v in s.voxel]
    c = [-1.0 + (torch.arange(d, device=DEV).double() + 0.5) * v for d, v in zip(s.dims, h)]
    out, size = torch.zeros(s.dims[::-1], device=DEV, dtype=torch.float64), 16
    for k in range(0, s.dims[2], size):
        z = c[2][k:k + size]
        in_z = ((mu - half)[:, 2] <= z[-1]) & ((mu + half)[:, 2] >= z[0])
        near = [v[in_z] for v in (mu, half, P, kap)]
        for j in range(0, s.dims[1], size):
            y = c[1][j:j + size]
            in_y = ((near[0] - near[1])[:, 1] <= y[-1]) & ((near[0] + near[1])[:, 1] >= y[0])
            row = [v[in_y] for v in near]
            for i in range(0, s.dims[0], size):
                x = c[0][i:i + size]
                sel = ((row[0] - row[1])[:, 0] <= x[-1]) & ((row[0] + row[1])[:, 0] >= x[0])
                m, _, Q, kk = (v[sel] for v in row)
                dx, dy, dz = (a[None, :] - m[:, b:b + 1] for a, b in ((x, 0), (y, 1), (z, 2)))
                e = (torch.log(kk)[:, None] - 0.5 * Q[:, 0, 0, None] * dx * dx)[:, None, None, :]
                e = e - 0.5 * (Q[:, 1, 1, None] * dy * dy)[:, None, :, None]
                e = e - (Q[:, 0, 1, None, None] * dy[:, :, None] * dx[:, None, :])[:, None]
                e = e - 0.5 * (Q[:, 2, 2, None] * dz * dz)[:, :, None, None]
                e = e - dz[:, :, None, None] * (Q[:, 0, 2, None, None] * dx[:, None, :] +
                                                Q[:, 1, 2, None, None] * dy[:, :, None])[:, None]
                out[k:k + size, j:j + size, i:i + size] = torch.exp(e).sum(0)
    return [out]


def exact(case, seed):
    """run()'s outputs in 64 bits; None for the cases whose sums would take too long that way.  Sums run over
    every pair that can reach the cut-off, footprints a little larger than the package's own."""
    k, n = case["kind"], case["n"]
    if k == "tomo_step" or (k not in ("tomo", "cone", "voxel") and n * case["views"] > 200000):
        return None
    s = _inputs(case, seed)
    p = [v.double() for v in s.params]
    if k == "tomo":
        return _exact_tomo(s, p)
    if k == "voxel":
        return _exact_voxel(s, p)
    if k == "cone":
        _, T, grads = _exact_views(s, p, "exact", TAU_CUT, True, cone=True)
        return [T, *grads]
    mode = case["mode"]
    cut = TAU_CUT if mode == "exact" else 1.0 / 255.0 if mode == "splat" else -math.log1p(-1.0 / 255.0)
    rgb, T, grads = _exact_views(s, p, mode, cut, k in ("train", "train_ws"))
    if k == "frame":
        return [rgb, T]
    if k == "march":
        return [rgb, T, *_exact_march(s, p, rgb)]
    if k == "train_ws":
        return [rgb, T, s.scale * ((rgb - s.target.double()) ** 2).sum().reshape(1), *grads]
    return [rgb, T, *grads]
