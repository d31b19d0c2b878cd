"""The grid-wide depth sort puts culled Gaussians behind the others and sorts the visible ones only, by buckets between sampled
keys; where the camera's near plane lets depths be zero or negative all are sorted together, digit by digit.  The order and
the lists must be the same, whatever share is culled and however the depths are spread."""
import dataclasses

import numpy as np
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


def _scene_at(depths, seed):
    sc = scenes.box_scene(len(depths), 2.0, 3.0, 4.0, -4.0, 0.5, 1.0, scenes.APP_SH, seed=seed)
    means = sc.means.copy()
    means[:, 2] = depths
    return dataclasses.replace(sc, means=means)


@pytest.mark.parametrize("kind", ["planes", "plane_and_box", "far_outliers", "samples_culled", "falling"])
@pytest.mark.parametrize("n", [12_000, 60_001, 600_000])                     # 600 000: buckets of 2048 and more
def test_depths_that_do_not_spread(kind, n):
    rng = np.random.default_rng(n)
    if kind == "planes":                                                  # crowded bins in the sample and in buckets between two
        depths = rng.choice([2.5, 3.0, 6.0], n)
    elif kind == "plane_and_box":
        depths = np.where(rng.random(n) < 0.5, 3.0, rng.uniform(2.0, 8.0, n))
    elif kind == "far_outliers":
        depths = np.where(rng.random(n) < 0.001, 90.0, 3.0 + 1e-5 * rng.random(n))
    elif kind == "falling":                                               # neighbours in memory in one bucket
        depths = np.linspace(8.0, 2.0, n)
    else:                                                                 # no sample is visible: one bucket holds them all
        stride = min(2048, max(256, n // 148)) // 8
        j = np.arange((n + stride - 1) // stride, dtype=np.uint64)
        at = j * np.uint64(stride) + ((j * np.uint64(2654435761) & np.uint64(0xffffffff)) * np.uint64(stride) >> np.uint64(32))
        depths = rng.uniform(2.0, 8.0, n)
        depths[at[at < n].astype(np.int64)] = -5.0
        if n > 60001:
            depths[40000:] = -5.0
    gpu = _check(_scene_at(depths.astype(np.float32), n), scenes.identity_camera(333, 217, 300.0))
    if kind == "samples_culled":
        assert gpu.visible.sum() > 8192          # beyond a CTA's shared memory


@pytest.mark.parametrize("n", [4_194_304, 4_194_305])                     # the largest scene for buckets, the smallest beyond
def test_line_between_buckets_and_digits(n):
    _check(scenes.box_scene(n, 3.0, -6.0, 8.0, -6.0, 0.5, 1.0, scenes.APP_NEURAL, seed=7), scenes.identity_camera(333, 217, 300.0))
