"""The grid-wide depth sort puts culled Gaussians behind the others in its first pass and sorts the visible ones only; where
the camera's near plane lets depths be zero or negative they are sorted together.  Up to 148 blocks of 1024 Gaussians each
pass also counts the next one's digits.  The order and the lists must be the same, whatever share is culled."""
import dataclasses

import pytest

from paper_2609_05255_b200 import scenes
from test_gpu_bin_cluster import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("near", [0.2, 0.0, -2.5])
@pytest.mark.parametrize("n,z_lo", [(32769, 2.0), (40001, -6.0), (33000, -300.0), (151552, -6.0), (151553, -6.0)])  # none, half, nearly all culled; block limit
def test_order_with_culled_gaussians(n, z_lo, near):
    sc = scenes.box_scene(n, 3.0, z_lo, 8.0, -3.5, 0.8, 1.0, scenes.APP_SH, seed=n)
    cam = dataclasses.replace(scenes.identity_camera(333, 217, 300.0), near_plane=near)
    gpu = _check(sc, cam)
    if z_lo > 0 and near > 0:
        assert gpu.visible.mean() > 0.3
