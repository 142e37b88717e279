"""The ray march's passes of 16 samples split over groups of CTAs (no early stop) against the same
passes in sequence, and against the FP64 oracle, at sample counts around the pass size.

T_stop = 1e-30 never ends a pixel of these scenes but selects the sequential form; the two forms
round the same sums in another order: at most 64 groups, so 64 x 2^-24 relative on colours of at most
about 4, i.e. below 2e-5."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import flat, run_forward

pytestmark = pytest.mark.gpu


def _march(ws, P, n, raster=None):
    import torch

    rgb, T = torch.full((P, 3), float("nan"), device="cuda:0"), torch.full((P,), float("nan"), device="cuda:0")
    err = None if raster is None else torch.full((P,), float("nan"), device="cuda:0")
    ws.ray_march(1.5, 7.0, n, rgb, T, raster, err)
    return rgb.double().cpu().numpy(), T.double().cpu().numpy(), None if err is None else err.double().cpu().numpy()


@pytest.mark.parametrize("n_samples", [1, 15, 16, 17, 161, 300, 2500])
def test_groups_match_sequence(gpu_lib, n_samples):
    import torch

    vg = gpu_lib
    sc = synth.uniform_scene(400, 65, log_scale=(-3.9, -2.3), kappa=(0.5, 20.0), sh_degree=1, sh_std=0.3, extent=0.8)
    cams = [synth.look_at((0.3, -0.4, -4.0), (0, 0, 0), 53, 37, 50.0), synth.look_at((-3.5, 0.5, 1.0), (0, 0, 0), 17, 64, 45.0)]
    o = dict(oracle.EXACT, bg=(0.2, 0.1, 0.4))
    ws, _, raster, _ = run_forward(vg, sc, cams, o)
    P = raster.shape[0]
    r = torch.as_tensor(np.ascontiguousarray(raster, np.float32)).to("cuda:0")
    a = _march(ws, P, n_samples, r)
    ws1, _, _, _ = run_forward(vg, sc, cams, dict(o, T_stop=1e-30))
    b = _march(ws1, P, n_samples, r)
    for x, y in zip(a, b):
        assert np.max(np.abs(x - y)) < 2e-5
    ref_rgb, ref_T = oracle.ray_march(sc, cams, o, 1.5, 7.0, n_samples)
    if n_samples >= 161:   # 30 samples a unit: the narrowest Gaussian (0.02) spans a sample spacing
        assert np.max(np.abs(a[0] - flat(ref_rgb))) < 1e-4
        assert np.max(np.abs(a[1] - flat(ref_T))) < 1e-4


def test_fixed_capacity_keeps_accepting(gpu_lib):
    """A fixed-capacity workspace marches whatever its partial results' buffer holds: more samples, larger views."""
    vg = gpu_lib
    sc = synth.uniform_scene(100, 66, log_scale=(-3.9, -2.3), kappa=(0.5, 20.0), sh_degree=0, sh_std=0.3, extent=0.8)
    small, large = (synth.look_at((0.3, -0.4, -4.0), (0, 0, 0), w, w, 50.0) for w in (32, 96))
    free = {}
    for cam in (small, large):
        ws, _, raster, _ = run_forward(vg, sc, [cam], oracle.EXACT)
        free[cam.width] = _march(ws, raster.shape[0], 200)
    ws = vg.Workspace()
    ws.reserve(100, 100000, 96 * 96, 36)
    for cam, n in ((large, 0), (small, 16), (small, 200), (large, 200)):
        ws, _, raster, _ = run_forward(vg, sc, [cam], oracle.EXACT, ws=ws, flags=vg.FLAG_FIXED_CAPACITY)
        if n == 0:   # the views' own buffers at their largest
            continue
        got = _march(ws, raster.shape[0], n)
        if n == 200:
            for x, y in zip(got[:2], free[cam.width][:2]):
                assert np.max(np.abs(x - y)) < 2e-5
