"""The forward's forms around their limits: one pixel per thread up to 2,432 tiles, two CTAs per tile up to
1,216, lists of any length modulo the records evaluated together.  Every pixel is evaluated by the
same operations in all of them, so images, transmittances and replay states are equal bit for bit."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import run_forward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 5, 400])
@pytest.mark.parametrize("mode", ["exact", "compat", "splat"])
@pytest.mark.parametrize("w,h,tile", [(16, 16, (0, 0)), (37, 21, (16, 8)), (70, 33, (32, 16)), (608, 512, (0, 0)),
                                      (624, 512, (0, 0)), (1024, 608, (0, 0)), (1040, 608, (0, 0))])
def test_forms_give_the_same_bits(gpu_lib, n, mode, w, h, tile):
    if n != 400 and w > 70:
        return   # short lists: the small images suffice
    vg = gpu_lib
    sc = synth.uniform_scene(n, 31 + n, log_scale=(-3.5, -2.0), kappa=(0.5, 20.0), sh_degree=1, sh_std=0.3, extent=0.6)
    if mode == "splat":
        sc.kappa = np.random.default_rng(7).uniform(0.05, 0.95, n).astype(np.float32)
    o = dict(oracle.EXACT if mode == "exact" else oracle.COMPAT, bg=(0.1, 0.2, 0.3), splat=mode == "splat")
    cam = synth.look_at((0.2, -0.3, -3.0), (0, 0, 0), w, h, 50.0)
    ref = None
    for ppt in (0, 1, 2, 4):
        ws, _, rgb, T = run_forward(vg, sc, [cam], o, ppt=ppt, tile=tile)
        S, last = ws.read_pixel_state()
        got = (rgb, T, S, last)
        assert ref is None or all(np.array_equal(a, b) for a, b in zip(ref, got)), ppt
        ref = ref or got
