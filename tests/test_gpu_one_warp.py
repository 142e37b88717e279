"""Images that one warp covers (8 x 4 pixels or fewer): a Gaussian's gradient sums then take one reduction per view, in one
order, so equal arithmetic gives equal bits.  On larger images the order in which the warps' sums arrive differs from run
to run, and the scale gradients of strongly flattened Gaussians show it (1e-5 of their norm and more between two runs of
one build), which hides whether two kernels round alike.  Here they must: repeated runs, and 16-bit SH rows read in
16-byte pieces, element by element (an array that is not 16-byte aligned) or widened to FP32 beforehand."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rec", ["float32", "bfloat16"])
@pytest.mark.parametrize("size", [(1, 1), (8, 4)])
def test_equal_bits(gpu_lib, size, rec):
    import torch

    vg = gpu_lib
    n, dt = 4000, getattr(torch, rec)
    sc = synth.uniform_scene(n, 611, log_scale=(-4.0, -2.0), sh_degree=3, sh_std=0.3, extent=0.9)
    scale = sc.scale.copy()
    scale[np.arange(0, n, 3), np.arange(0, n, 3) % 2] /= 100.0   # flattened 100:1
    cams = [synth.look_at(eye, (0, 0, 0), *size, 2.0) for eye in ((0.1, -4.0, 0.2), (3.0, 2.0, -2.0), (-3.5, 0.5, 1.5))]
    P = sum(c.width * c.height for c in cams)
    t = lambda a, d=torch.float32: torch.tensor(a, device="cuda:0").to(d)
    sh16 = t(sc.sh, torch.float16)
    off = torch.empty(sh16.numel() + 1, device="cuda:0", dtype=torch.float16)[1:].view(sh16.shape).copy_(sh16)
    w = torch.randn((P, 3), device="cuda:0", generator=torch.Generator("cuda:0").manual_seed(4))
    out = []
    for sh in (sh16, sh16, off, sh16.float()):
        ws = vg.Workspace()
        g = vg.Gaussians(t(sc.mu), t(scale, dt), t(sc.quat, dt), t(sc.kappa, dt), sh, 3)
        rgb = torch.empty((P, 3), device="cuda:0")
        grads = [torch.zeros(s, device="cuda:0") for s in ((n, 3), (n, 3), (n, 4), (n,), (n, 16, 3))]
        ws.preprocess(g, cams, vg.Opts.compat())
        ws.bin_sort()
        ws.render_fwd(rgb)
        ws.render_bwd(w, None, *grads)
        out.append([rgb, *grads])
    assert int((out[0][2] != 0).sum()) > 100
    for other in out[1:]:
        for a, b in zip(other, out[0]):
            assert torch.equal(a, b)
