"""Binning of few items by one CTA (up to 4,096) and of more by the radix passes: lists bit-exact against the
oracle at the sizes where the one-CTA form changes, with many equal depths, and when the instance
buffers grow, shrink or are fixed from call to call."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import dev_scene, vg_opts

pytestmark = pytest.mark.gpu


def _check(vg, ws, scene, cams, flags=0):
    o = dict(oracle.COMPAT)
    ws.preprocess(dev_scene(vg, scene), cams, vg_opts(vg, o, flags))
    ws.bin_sort()
    L = oracle.lists(scene, cams, o)
    ts, items = ws.read_bins()
    assert np.array_equal(ts, L["tile_start"])
    v = np.concatenate([np.repeat(k, c) for k, c in enumerate(np.diff(np.asarray(L["tile_start"])[np.append(L["tile_base"][:len(cams)], len(ts) - 1)]))])
    assert np.array_equal(items - v * scene.n, L["sorted_g"])


def _scene(n, seed, planes=0):
    sc = synth.uniform_scene(n, seed, log_scale=(-4.5, -3.5), kappa=(0.5, 20.0), sh_degree=0, sh_std=0.3, extent=0.8)
    if planes:   # equal depths: ties keep the items' order
        sc.mu[:, 2] = np.float32(0.1) * (np.arange(n) % planes)
    return sc


@pytest.mark.parametrize("n", [1, 2, 31, 33, 512, 513, 2047, 2048, 2049, 4095, 4096, 4097, 12289])
@pytest.mark.parametrize("planes", [0, 1, 3])
def test_lists_at_size_limits(gpu_lib, n, planes):
    vg = gpu_lib
    _check(vg, vg.Workspace(), _scene(n, 300 + n, planes), [synth.look_at((0.0, 0.0, -4.0), (0, 0, 0), 64, 48, 50.0)])


def test_one_workspace_over_sizes(gpu_lib):
    vg = gpu_lib
    ws = vg.Workspace()
    one = [synth.look_at((0.0, 0.0, -4.0), (0, 0, 0), 64, 48, 50.0)]
    two = one + [synth.look_at((0.5, -3.0, 1.0), (0, 0, 0), 33, 80, 45.0)]
    for n, cams in ((40, one), (5000, two), (300, one), (9000, two), (20000, one), (40, two)):
        _check(vg, ws, _scene(n, 400 + n), cams)
    for n, cams in ((9000, two), (40, one), (20000, one)):
        _check(vg, ws, _scene(n, 400 + n), cams, flags=vg.FLAG_FIXED_CAPACITY)


@pytest.mark.parametrize("n", [300, 20000])
def test_fixed_capacity_captured_after_a_plain_binning(gpu_lib, n):
    """A step with a fixed capacity captured right after one plain step (nothing reserved): the scratch is there."""
    import torch

    vg = gpu_lib
    sc, cam = _scene(n, 500 + n), [synth.look_at((0.0, 0.0, -4.0), (0, 0, 0), 64, 48, 50.0)]
    g, ws = dev_scene(vg, sc), vg.Workspace()
    out = torch.empty((64 * 48, 3), device="cuda:0")

    def step(flags):
        ws.preprocess(g, cam, vg_opts(vg, dict(oracle.COMPAT), flags))
        ws.bin_sort()
        ws.render_fwd(out)

    step(0)
    want = out.clone()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step(vg.FLAG_FIXED_CAPACITY)
    for _ in range(2):
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want)
