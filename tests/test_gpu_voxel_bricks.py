"""The voxel query at the edges of its bricks (8^3), half bricks (8 x 4 x 4) and chunks of 64 records, against
the FP64 oracle.  A sigma_cut of 0.05 makes the boxes visible in the values.  Sums of at most ~300
FP32 terms: 1e-4 of the largest value, as in the voxel tests."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import dev_scene, vg_opts

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 63, 64, 65, 129, 300])
@pytest.mark.parametrize("dims", [(1, 1, 1), (8, 8, 8), (9, 4, 5), (3, 17, 12), (40, 23, 16), (7, 5, 33)])
def test_voxel_bricks(gpu_lib, n, dims):
    import torch

    vg = gpu_lib
    scene = synth.tomo_scene(n, 140 + n, log_scale=(-3.5, -1.0))
    origin, voxel = (-1.0, -0.9, -0.8), tuple(1.9 / d for d in dims)
    out = torch.full(dims[::-1], float("nan"), device="cuda:0")
    o = dict(oracle.EXACT, tau_cut=0.05)
    vg.Workspace().query_density(dev_scene(vg, scene), origin, voxel, dims, vg_opts(vg, o), out)
    got = out.cpu().numpy().astype(np.float64)
    ref = oracle.voxel_density(scene, origin, voxel, dims, sigma_cut=0.05)
    assert np.max(np.abs(got - ref)) <= 1e-4 * max(np.max(np.abs(ref)), 1e-30)
