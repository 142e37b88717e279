"""The cone beam's backward per (view, Gaussian) at the edges of its strips (4 to 32 lanes side by side, two
rows a lane), against the FP64 oracle, and where it gives way to the blend's backward (counted pairs,
a fixed-capacity workspace whose weights' buffer is too small).  Gradients within 1e-3 of each Gaussian's block,
as in the cone tests."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import check_grads, dev_scene, vg_opts

pytestmark = pytest.mark.gpu


def _run(vg, scene, cams, dL, ws=None, flags=0):
    import torch

    n, P = scene.n, sum(c.width * c.height for c in cams)
    proj = torch.full((P,), float("nan"), device="cuda:0")
    grads = [torch.zeros(s, device="cuda:0") for s in ((n, 3), (n, 3), (n, 4), (n,))]
    ws = ws or vg.Workspace()
    ws.project_cone(dev_scene(vg, scene), cams, vg_opts(vg, oracle.EXACT, flags), proj,
                    torch.as_tensor(dL.astype(np.float32)).to("cuda:0"), *grads)
    return proj.double().cpu().numpy(), {k: t.double().cpu().numpy() for k, t in zip(("mu", "scale", "quat", "kappa"), grads)}


def _ref(scene, cams, dL):
    L = oracle.lists(scene, cams, oracle.EXACT)
    split = np.cumsum([0] + [c.width * c.height for c in cams])
    return oracle.cone_grad(scene, cams, oracle.EXACT, L, [dL[split[v]:split[v + 1]] for v in range(len(cams))])


@pytest.mark.parametrize("n", [1, 40, 3000])
@pytest.mark.parametrize("sizes", [[(1, 1)], [(5, 70), (33, 9)], [(130, 41)], [(64, 64), (3, 3), (17, 31)]])
def test_cone_backward_sizes(gpu_lib, n, sizes):
    vg = gpu_lib
    scene = synth.tomo_scene(n, 201, log_scale=(-4.5, -2.0))
    cams = [synth.look_at((0.5 + v, -3.0, 1.0 - v), (0, 0, 0), w, h, 45.0) for v, (w, h) in enumerate(sizes)]
    dL = np.random.default_rng(5).normal(size=sum(w * h for w, h in sizes))
    proj, g = _run(vg, scene, cams, dL)
    ref = _ref(scene, cams, dL)
    counted, gc = _run(vg, scene, cams, dL, flags=vg.FLAG_COUNT_PAIRS)
    assert np.array_equal(proj, counted)
    for grads in (g, gc):
        if all(not ref[k].any() for k in grads):   # the Gaussian lies outside every view
            assert all(not grads[k].any() for k in grads)
        else:
            check_grads(grads, ref, scene, 1e-3, keys=("mu", "scale", "quat", "kappa"))


def test_fixed_capacity_keeps_accepting(gpu_lib):
    vg = gpu_lib
    scene = synth.tomo_scene(50, 202, log_scale=(-4.0, -2.5))
    small, large = ([synth.look_at((0.5, -3.0, 1.0), (0, 0, 0), w, w, 45.0)] for w in (16, 64))
    dL = np.random.default_rng(6).normal(size=64 * 64)
    ws = vg.Workspace()
    ws.reserve(50, 100000, 64 * 64, 16)
    ws.project_cone(dev_scene(vg, scene), large, vg_opts(vg, oracle.EXACT, vg.FLAG_FIXED_CAPACITY),
                    __import__("torch").empty(64 * 64, device="cuda:0"))   # the views' own buffers at their largest
    for cams, d in ((small, dL[:256]), (large, dL)):
        _, g = _run(vg, scene, cams, d, ws=ws, flags=vg.FLAG_FIXED_CAPACITY)
        check_grads(g, _ref(scene, cams, d), scene, 1e-3, keys=("mu", "scale", "quat", "kappa"))
