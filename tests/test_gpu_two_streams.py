"""The two backwards of one forward, vg_render_bwd and vg_render_bwd_noalloc, on two streams at once: neither writes what the
other reads.  Gradients as of the one alone, up to the order of the warps' sums (1e-5 of the largest)."""
import pytest

import synth
from gpu_util import dev_scene

pytestmark = pytest.mark.gpu


def test_two_backwards_at_once(gpu_lib):
    import torch

    vg = gpu_lib
    scene = synth.uniform_scene(3000, 301, log_scale=(-4.0, -2.5), sh_degree=1, sh_std=0.3, extent=0.9)
    cams = synth.small_views(2, 5, [(330, 210), (150, 90)])
    P = sum(c.width * c.height for c in cams)
    g, ws = dev_scene(vg, scene), vg.Workspace()
    new = lambda: [torch.zeros(s, device="cuda:0") for s in ((g.n, 3), (g.n, 3), (g.n, 4), (g.n,), (g.n, 4, 3))]
    w, want = torch.randn((P, 3), device="cuda:0"), new()
    streams = [torch.cuda.Stream() for _ in range(2)]
    for _ in range(10):
        got = [new(), new()]
        ws.preprocess(g, cams, vg.Opts.exact())
        ws.bin_sort()
        ws.render_fwd(torch.empty((P, 3), device="cuda:0"))
        torch.cuda.synchronize()
        ws.render_bwd_noalloc(w, None, *got[0], stream=streams[0])
        ws.render_bwd(w, None, *got[1], stream=streams[1])
        torch.cuda.synchronize()
        if not want[0].any():
            ws.render_bwd(w, None, *want)
        for grads in got:
            for x, y in zip(grads, want):
                assert float((x - y).abs().max()) <= 1e-5 * float(y.abs().max())
