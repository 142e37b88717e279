"""A pixel whose dL/dproj is not finite reaches the gradients of the Gaussians whose footprint holds it, and no others --
also not those whose footprint ends in the same group of eight columns.  One angle: every gradient is one sum, so the
untouched ones keep their bits.  Which footprints hold the pixel shows with dL/dproj = 1e30 there: round Gaussians have
tau >= 1e-14 on their whole rectangle (at its corners exp(-m^2 / 2) is the square of what it is at its sides)."""
import pytest

import synth
from gpu_util import dev_scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("at", [(0, 0), (20, 27), (20, 28), (33, 44)])
def test_untouched_gradients_stay(gpu_lib, at, bad):
    import torch

    vg = gpu_lib
    scene = synth.tomo_scene(400, 241, log_scale=(-4.5, -3.0))
    scene.scale[:] = scene.scale[:, :1]
    g = dev_scene(vg, scene)
    beam = synth.parallel_beam(1, det=45, extent=2.0)
    gen = torch.Generator("cuda:0").manual_seed(5)
    dL, out = torch.rand((1, 45, 45), device="cuda:0", generator=gen) + 0.5, []
    for value in (0.0, 1e30, bad):
        dL[0, at[0], at[1]] = value
        grads = [torch.zeros(s, device="cuda:0") for s in ((g.n, 3), (g.n, 3), (g.n, 4), (g.n,))]
        vg.Workspace().project_tomo(g, beam, vg.Opts(tau_cut=1e-6), torch.empty_like(dL), dL, *grads)
        out.append(torch.cat([t.reshape(g.n, -1) for t in grads], 1))
    zero, one, got = out
    untouched = (zero == one).all(1)
    assert untouched.sum() > 200
    assert torch.equal(got[untouched], zero[untouched])
    if at[0] == 20:   # pixels inside the ball
        assert (~untouched).any() and not torch.isfinite(got[~untouched]).all()
