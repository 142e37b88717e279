"""The autograd wrappers where they take a shorter way: the tomography backward with the forward's
projection and lists (and without, once a parameter, the geometry or the workspace changed), the
rasterizer's backward into buffers it does not clear and with an unused output.  Gradients equal those of
the library's own two calls up to the order of the sums over angles or warps (1e-5 of the largest)."""
import numpy as np
import pytest

import synth
from gpu_util import dev_scene

pytestmark = pytest.mark.gpu


def _leaves(scene):
    import torch
    return [torch.tensor(a, device="cuda:0", requires_grad=True) for a in (scene.mu, scene.scale, scene.quat, scene.kappa)]


def _direct(vg, params, beam, dL):
    import torch
    g = vg.Gaussians(*(p.detach().clone() for p in params), None, 0)
    proj = torch.empty((len(beam.angles), beam.det_h, beam.det_w), device="cuda:0")
    grads = [torch.zeros(p.shape, device="cuda:0") for p in params]
    ws = vg.Workspace()
    ws.project_tomo(g, beam, vg.Opts(tau_cut=1e-6), proj, dL, *grads)
    return proj, grads, ws.read_bins()


def _same(a, b):
    for x, y in zip(a, b):
        assert float((x - y).abs().max()) <= 1e-5 * float(y.abs().max())


@pytest.mark.parametrize("det", [32, 220])
@pytest.mark.parametrize("between", ["nothing", "proj", "param", "geometry", "other call", "twice"])
def test_tomo_backward_reuse(gpu_lib, det, between):
    import torch
    vg = gpu_lib
    scene = synth.tomo_scene(300, 210)
    beam = synth.parallel_beam(5, det=det, extent=2.0)
    params, pro = _leaves(scene), vg.Projector()
    dL = torch.rand((5, det, det), device="cuda:0", generator=torch.Generator("cuda:0").manual_seed(2))
    proj = pro.parallel(*params, beam)
    total = (proj * dL).sum()
    if between == "proj":
        proj.data.zero_()
    elif between == "param":
        with torch.no_grad():
            params[0].mul_(0.9)
    elif between == "geometry":
        beam.u0 += 0.05
    elif between == "other call":
        pro.parallel(*_leaves(synth.tomo_scene(40, 211)), synth.parallel_beam(3, det=16, extent=2.0))
    got = torch.autograd.grad(total, params, retain_graph=True)
    if between == "twice":
        got = torch.autograd.grad(total, params)
    _, want, (ts, items) = _direct(vg, params, beam, dL)
    _same(got, want)
    ts2, items2 = pro.ws.read_bins()
    assert np.array_equal(ts, ts2) and np.array_equal(items, items2)


@pytest.mark.parametrize("use", ["rgb", "T", "both"])
def test_render_backward_unused_outputs(gpu_lib, use):
    import torch
    vg = gpu_lib
    scene = synth.uniform_scene(200, 212, log_scale=(-3.5, -2.5), sh_degree=1, sh_std=0.3, extent=0.9)
    cams = synth.small_views(2, 3, [(40, 24), (31, 29)])
    P = sum(c.width * c.height for c in cams)
    w = torch.randn((P, 3), device="cuda:0") if use != "T" else torch.zeros((P, 3), device="cuda:0")
    v = torch.randn((P,), device="cuda:0") if use != "rgb" else torch.zeros((P,), device="cuda:0")
    leaves = _leaves(scene) + [torch.tensor(scene.sh, device="cuda:0", requires_grad=True)]
    junk = [torch.full(p.shape, float("nan"), device="cuda:0") for p in leaves]   # freed blocks the backward may get
    del junk
    rgb, T = vg.Rasterizer(vg.Opts.exact()).render(*leaves, cams)
    loss = {"rgb": lambda: (rgb * w).sum(), "T": lambda: (T * v).sum(), "both": lambda: (rgb * w).sum() + (T * v).sum()}[use]()
    got = torch.autograd.grad(loss, leaves)
    ws = vg.Workspace()
    want = [torch.zeros(p.shape, device="cuda:0") for p in leaves]
    ws.preprocess(dev_scene(vg, scene), cams, vg.Opts.exact())
    ws.bin_sort()
    ws.render_fwd(torch.empty((P, 3), device="cuda:0"))
    ws.render_bwd(w, v, *want)
    for x, y in zip(got, want):
        assert torch.isfinite(x).all()
        assert float((x - y).abs().max()) <= 1e-5 * max(float(y.abs().max()), 1e-30)
