"""A fixed-capacity cone-beam gradient captured right after a reservation (the camera table aside, which a projection uploads)
takes the item-wise backward: it makes the launches of an eager call, one fewer than the blend's backward, and the replay
leaves the gradients of an eager call, up to the order of the sums over views (1e-5 of the largest)."""
import pytest

import synth
from gpu_util import dev_scene

pytestmark = pytest.mark.gpu


def test_captured_right_after_a_reservation(gpu_lib):
    import torch

    vg = gpu_lib
    g = dev_scene(vg, synth.tomo_scene(200, 271))
    cams = [synth.look_at(eye, (0, 0, 0), w, h, 45.0) for eye, w, h in (((0.5, -3.0, 1.0), 70, 41), ((3.0, 0.2, -1.0), 33, 64))]
    P, tiles = sum(c.width * c.height for c in cams), sum((c.width + 15) // 16 * ((c.height + 15) // 16) for c in cams)
    o = vg.Opts(tau_cut=1e-6, flags=vg.FLAG_FIXED_CAPACITY | vg.FLAG_GRAD_ZERO)
    proj, dL = torch.empty(P, device="cuda:0"), torch.randn(P, device="cuda:0")
    new = lambda: [torch.zeros(s, device="cuda:0") for s in ((g.n, 3), (g.n, 3), (g.n, 4), (g.n,))]
    ws, got, want = vg.Workspace(), new(), new()
    ws.reserve(2 * g.n, 100000, P, tiles)
    ws.project_cone(g, cams, o, proj)
    torch.cuda.synchronize()
    launches, graph = ws.query()["launches"], torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ws.project_cone(g, cams, o, proj, dL, *got)
    captured = ws.query()["launches"] - launches
    graph.replay()
    torch.cuda.synchronize()
    eager = vg.Workspace()
    eager.project_cone(g, cams, vg.Opts(tau_cut=1e-6, flags=vg.FLAG_GRAD_ZERO), torch.empty_like(proj))
    launches = eager.query()["launches"]
    eager.reserve(2 * g.n, 100000, P, tiles)
    eager.project_cone(g, cams, o, proj, dL, *want)
    assert captured == eager.query()["launches"] - launches
    for x, y in zip(got, want):
        assert float((x - y).abs().max()) <= 1e-5 * float(y.abs().max())
