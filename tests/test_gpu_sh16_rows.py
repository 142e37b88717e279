"""Degree-3 SH rows in 16 bits read in 16-byte pieces, against the same values in FP32 (widening is exact, so images
are equal bit for bit and gradients up to the order of the warps' sums) and against an array that is not
16-byte aligned, which is read element by element; counts around a warp's 32 rows."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 32, 33, 95, 500])
@pytest.mark.parametrize("dtype", ["float16", "bfloat16"])
def test_sh16_rows(gpu_lib, n, dtype):
    import torch

    vg = gpu_lib
    dt = getattr(torch, dtype)
    sc = synth.uniform_scene(n, 500 + n, log_scale=(-3.0, -2.0), sh_degree=3, sh_std=0.3, extent=0.7)
    cams = synth.small_views(2, 3, [(40, 24), (31, 29)])
    P = sum(c.width * c.height for c in cams)
    t = lambda a: torch.tensor(a, device="cuda:0")
    sh16 = t(sc.sh).to(dt)
    off = torch.empty(sh16.numel() + 1, device="cuda:0", dtype=dt)[1:].view(sh16.shape).copy_(sh16)
    assert off.data_ptr() % 16 and sh16.data_ptr() % 16 == 0
    w, out = torch.randn((P, 3), device="cuda:0", generator=torch.Generator("cuda:0").manual_seed(3)), []
    for sh in (sh16.float(), sh16, off):
        ws = vg.Workspace()
        g = vg.Gaussians(t(sc.mu), t(sc.scale), t(sc.quat), t(sc.kappa), sh, 3)
        rgb = torch.empty((P, 3), device="cuda:0")
        grads = [torch.zeros(s, device="cuda:0") for s in ((n, 3), (n, 3), (n, 4), (n,), (n, 16, 3))]
        ws.preprocess(g, cams, vg.Opts.exact())
        ws.bin_sort()
        ws.render_fwd(rgb)
        ws.render_bwd(w, None, *grads)
        out.append((rgb, grads))
    for rgb, grads in out[1:]:
        assert torch.equal(rgb, out[0][0])
        for a, b in zip(grads, out[0][1]):
            assert float((a - b).abs().max()) <= 1e-5 * max(float(b.abs().max()), 1e-30)
