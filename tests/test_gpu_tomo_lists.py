"""The tomography's backward without lists (VG_FLAG_NO_LISTS) on another beam than the one whose lists the workspace holds:
the read-backs keep describing the call with lists, and the gradient is the one of the call with lists, up to the order of
the sums over angles (1e-5 of the largest)."""
import numpy as np
import pytest

import synth
from gpu_util import dev_scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first,second", [((3, 16), (5, 240)), ((5, 240), (3, 16)), ((4, 64), (4, 64))])
def test_read_backs_keep_the_lists(gpu_lib, first, second):
    import torch

    vg = gpu_lib
    few, many = (dev_scene(vg, synth.tomo_scene(n, 231)) for n in (40, 300))
    beams = [synth.parallel_beam(a, det=d, extent=2.0) for a, d in (first, second)]
    g0, g1 = (few, many) if first[1] < second[1] else (many, few)
    new = lambda b: torch.empty((len(b.angles), b.det_h, b.det_w), device="cuda:0")
    grads = lambda g: [torch.zeros(s, device="cuda:0") for s in ((g.n, 3), (g.n, 3), (g.n, 4), (g.n,))]
    ws = vg.Workspace()
    ws.project_tomo(g0, beams[0], vg.Opts(tau_cut=1e-6), new(beams[0]))
    q, bins, keys = ws.query(), ws.read_bins(), ws.read_keys()
    other = vg.Workspace()
    proj, want, got = new(beams[1]), grads(g1), grads(g1)
    other.project_tomo(g1, beams[1], vg.Opts(tau_cut=1e-6), proj)
    dL = torch.rand(proj.shape, device="cuda:0", generator=torch.Generator("cuda:0").manual_seed(3))
    other.project_tomo(g1, beams[1], vg.Opts(tau_cut=1e-6, flags=vg.FLAG_PROJ_GIVEN), proj, dL, *want)
    ws.project_tomo(g1, beams[1], vg.Opts(tau_cut=1e-6, flags=vg.FLAG_PROJ_GIVEN | vg.FLAG_NO_LISTS), proj, dL, *got)
    for x, y in zip(got, want):
        assert float((x - y).abs().max()) <= 1e-5 * float(y.abs().max())
    q2 = ws.query()
    assert all(q[k] == q2[k] for k in ("n_items", "n_instances", "n_tiles", "n_pixels"))
    for a, b in zip(bins + keys, ws.read_bins() + ws.read_keys()):
        assert np.array_equal(a, b)
    counts, items = ws.read_bins_range(0, q["n_tiles"], q["n_instances"])
    assert np.array_equal(np.cumsum(counts), bins[0][1:]) and np.array_equal(items, bins[1])
