"""Tomography kernels at the edges of their tiles, rows and item batches, against the FP64 oracle.

The projector owns 2 x 4 pixels per lane of 16 x 16 tiles; the backward walks each item's pixel
rectangle in columns of 8 (1, 2 or 4 lanes side by side), takes several items per warp once there are
enough, and orders the items by tile once a view's weights exceed 160 KB.  The bars are those of the
tomography tests: projections within 1e-4, gradients within 1e-3 of each Gaussian's block (FP32 sums
of at most ~1e5 pixels against FP64)."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import dev_scene, grad_block_err

pytestmark = pytest.mark.gpu


def _beam(angles, w, h, extent):
    b = synth.parallel_beam(angles, det=8, extent=extent)
    f = lambda x: float(np.float32(x))
    return synth.Beam(b.angles, w, h, f(extent / w), f(extent / h), f(-extent / 2), f(-extent / 2))


CASES = [(1, 1, 1, 3, 2.0), (1, 7, 5, 3, 2.0), (40, 8, 8, 3, 2.0), (40, 9, 17, 3, 1.0), (300, 33, 16, 2, 1.0),
         (300, 15, 50, 2, 2.0), (64, 250, 211, 2, 1.0), (6000, 24, 24, 20, 2.0)]


@pytest.mark.parametrize("n,w,h,angles,extent", CASES)
def test_tomo_sizes(gpu_lib, n, w, h, angles, extent):
    import torch

    vg = gpu_lib
    scene = synth.tomo_scene(n, 77)
    beam = _beam(angles, w, h, extent)
    rng = np.random.default_rng(3)
    dL = rng.normal(size=(angles, h, w))
    L = oracle.tomo_lists(scene, beam, 1e-6)
    _, ref = oracle.tomo(scene, beam, L)
    gref = oracle.tomo_grad(scene, beam, L, dL)
    ws, g = vg.Workspace(), dev_scene(vg, scene)
    proj = torch.full((angles, h, w), float("nan"), device="cuda:0")
    grads = [torch.full(s, float("nan"), device="cuda:0") for s in ((n, 3), (n, 3), (n, 4), (n,))]
    dLt = torch.as_tensor(dL.astype(np.float32)).to("cuda:0")
    ws.project_tomo(g, beam, vg.Opts(tau_cut=1e-6, flags=vg.FLAG_GRAD_ZERO), proj, dLt, *grads)
    assert np.max(np.abs(proj.cpu().numpy() - ref)) < 1e-4
    for k, t in zip(("mu", "scale", "quat", "kappa"), grads):
        if np.max(np.abs(gref[k])) > 0:
            e = grad_block_err(t.cpu().numpy(), gref[k], n)
            assert e.max() < 1e-3, (k, e.max())
    # the same walk without atomics between items: projections repeat bit for bit
    again = torch.empty_like(proj)
    ws.project_tomo(g, beam, vg.Opts(tau_cut=1e-6), again)
    assert torch.equal(proj, again)


@pytest.mark.parametrize("w,h", [(31, 18), (200, 220)])
def test_tomo_fused_loss_padded_rows(gpu_lib, w, h):
    """The fused step's pixel weights sit in padded rows: loss and gradients equal the two-call form's."""
    import torch

    vg = gpu_lib
    scene = synth.tomo_scene(200, 78)
    beam = _beam(3, w, h, 2.0)
    ws, g = vg.Workspace(), dev_scene(vg, scene)
    tgt = torch.rand((3, h, w), device="cuda:0", generator=torch.Generator("cuda:0").manual_seed(1))
    o = vg.Opts(tau_cut=1e-6, flags=vg.FLAG_GRAD_ZERO)
    mk = lambda: [torch.empty(s, device="cuda:0") for s in ((200, 3), (200, 3), (200, 4), (200,))]
    proj, loss, ga, gb = torch.empty_like(tgt), torch.empty(1, device="cuda:0"), mk(), mk()
    ws.tomo_l2_step(g, beam, o, tgt, 0.5, proj, loss, *ga)
    ws.project_tomo(g, beam, o, proj, (proj - tgt), *gb)
    d = (proj.double() - tgt.double())
    assert abs(float(loss) - float(0.5 * (d * d).sum())) < 1e-5 * float(0.5 * (d * d).sum())
    for a, b in zip(ga, gb):
        # sums over angles by atomics: a few ulp of each parameter's largest gradient
        assert float((a - b).abs().max()) <= 1e-5 * float(b.abs().max())
