"""The Python wrappers without a device: what they accept and what they hand to the library, with a stand-in for the
workspace where one is needed."""
from types import SimpleNamespace

import numpy as np
import pytest

import paper_2412_03378_gb300 as vg


@pytest.mark.parametrize("t", [[1.0, 2.0, 3.0], [1.0, 2.0, 3.0, 1.0], np.array([1.0, 2.0, 3.0, 1.0], np.float32)])
def test_camera_translation_may_be_homogeneous(t):
    """The first three entries of t are read, and the first nine of R."""
    cam = SimpleNamespace(R=np.eye(3), t=t, fx=10.0, fy=11.0, cx=2.0, cy=3.0, width=4, height=5)
    c = vg.camera_struct(cam)
    assert list(c.t) == [1.0, 2.0, 3.0] and list(c.R) == [1, 0, 0, 0, 1, 0, 0, 0, 1]
    cam.R = [[1, 0, 0], [0, 1, 0], [0, 0, 1], [7, 7, 7]]
    assert list(vg.camera_struct(cam).R) == [1, 0, 0, 0, 1, 0, 0, 0, 1]
