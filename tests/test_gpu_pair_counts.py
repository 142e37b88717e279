"""Where every footprint pixel counts, the pairs that a counted forward evaluates are those of the pixels still unfinished at
each record, whatever the pixels per thread and however many records are evaluated together."""
import pytest

import oracle
import synth
from gpu_util import run_forward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T_stop", [0.0, 0.05, 0.6])
def test_counts_do_not_depend_on_the_layout(gpu_lib, T_stop):
    vg = gpu_lib
    scene = synth.uniform_scene(1500, 291, log_scale=(-3.5, -2.0), kappa=(1.0, 40.0), extent=0.9)
    cams = synth.small_views(2, 4, [(75, 52), (40, 33)])
    counts = []
    for ppt in (1, 2, 4):
        ws, *_ = run_forward(vg, scene, cams, dict(oracle.EXACT, T_stop=T_stop), flags=vg.FLAG_COUNT_PAIRS, ppt=ppt)
        q = ws.query()
        counts.append((q["n_pairs"], q["n_blend"]))
    assert counts[0][0] > 10000 and counts[1] == counts[0] and counts[2] == counts[0]
