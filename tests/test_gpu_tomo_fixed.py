"""A fixed-capacity workspace takes the tomography's backward on a small detector and then on a larger one, in two calls and
fused, whether its buffer of pixel weights was reserved for the largest (as for a step of n_pixels and n_tiles) or is too
small for either, in which case the weights are formed where they are used.  Against a workspace that may grow: the
projections are equal, the gradients up to the order of the sums over angles (1e-5 of the largest)."""
import pytest

import synth
from gpu_util import dev_scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("reserved", [True, False])
@pytest.mark.parametrize("fused", [False, True])
def test_growing_detectors(gpu_lib, fused, reserved):
    import torch

    vg = gpu_lib
    g, A = dev_scene(vg, synth.tomo_scene(300, 261)), 4
    fixed = vg.Workspace()
    fixed.reserve(g.n * A, 400000, A * 230 * 230 if reserved else 30, A * 15 * 15)
    gen = torch.Generator("cuda:0").manual_seed(7)
    for det in (13, 45, 230):
        beam = synth.parallel_beam(A, det=det, extent=2.0)
        other = torch.rand((A, det, det), device="cuda:0", generator=gen)
        out = []
        for ws, flags in ((fixed, vg.FLAG_FIXED_CAPACITY), (vg.Workspace(), 0)):
            proj, loss = torch.empty_like(other), torch.empty(1, device="cuda:0")
            grads = [torch.zeros(s, device="cuda:0") for s in ((g.n, 3), (g.n, 3), (g.n, 4), (g.n,))]
            o = vg.Opts(tau_cut=1e-6, flags=flags)
            if fused:
                ws.tomo_l2_step(g, beam, o, other, 0.5, proj, loss, *grads)
            else:
                loss.zero_()
                ws.project_tomo(g, beam, o, proj)
                ws.project_tomo(g, beam, o, proj, other, *grads)
            out.append([proj, loss, *grads])
        assert torch.equal(out[0][0], out[1][0])
        for x, y in zip(out[0][1:], out[1][1:]):
            assert float((x - y).abs().max()) <= 1e-5 * float(y.abs().max())
