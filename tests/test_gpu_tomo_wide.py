"""Detectors up to 65,536 pixels wide or tall, against a detector of 512 that covers the same pixels; wider ones are refused
(a record holds a pixel coordinate in 16 bits).  The offset of a centre is a number near 65,536 there, rounded to 2^-8
pixels at worst, that is 2e-4 of the narrowest sigma (18 pixels), so projections and gradients agree within 2e-3 of the largest."""
from types import SimpleNamespace

import pytest

import synth
from gpu_util import dev_scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tall", [False, True])
def test_wide_detector(gpu_lib, tall):
    import torch

    vg = gpu_lib
    pitch, first, n = 1.0 / 1024, 65536 - 512, 512
    scene = synth.tomo_scene(30, 281, log_scale=(-4.0, -3.0), kappa=(0.5, 2.0))
    scene.mu[:] *= 0.2
    out = []
    for wide in (True, False):
        size = 65536 if wide else n
        start = -(first + n / 2) * pitch if wide else -n / 2 * pitch
        beam = SimpleNamespace(angles=[0.0, 0.7], det_w=1 if tall else size, det_h=size if tall else 1, pitch_u=pitch,
                               pitch_v=pitch, u0=0.0 if tall else start, v0=start if tall else 0.0)
        proj = torch.empty((2, beam.det_h, beam.det_w), device="cuda:0")
        dL = torch.zeros_like(proj)
        dL.view(2, -1)[:, -n:] = torch.rand((2, n), device="cuda:0", generator=torch.Generator("cuda:0").manual_seed(8))
        grads = [torch.zeros(s, device="cuda:0") for s in ((30, 3), (30, 3), (30, 4), (30,))]
        vg.Workspace().project_tomo(dev_scene(vg, scene), beam, vg.Opts(tau_cut=1e-6), proj, dL, *grads)
        out.append([proj.view(2, -1)[:, -n:], *grads])
    assert float(out[1][0].min()) < 0.9
    for x, y in zip(*out):
        assert float((x - y).abs().max()) <= 2e-3 * float(y.abs().max())


@pytest.mark.parametrize("w,h", [(65537, 1), (1, 65537), (70000, 1)])
def test_wider_is_refused(gpu_lib, w, h):
    import torch

    vg = gpu_lib
    beam = SimpleNamespace(angles=[0.0], det_w=w, det_h=h, pitch_u=0.1, pitch_v=0.1, u0=0.0, v0=0.0)
    with pytest.raises(vg.VGError) as e:
        vg.Workspace().project_tomo(dev_scene(vg, synth.tomo_scene(5, 282)), beam, vg.Opts(tau_cut=1e-6),
                                    torch.empty((1, h, w), device="cuda:0"))
    assert e.value.status == 1
