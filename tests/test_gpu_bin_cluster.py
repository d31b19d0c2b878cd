"""Binning of small scenes runs in one cluster of CTAs (up to 8192 Gaussians and 512 cells of 64 x 64 pixels), in which up
to 2048 Gaussians are ordered by counting and more by a radix sort; larger ones take the grid-wide kernels.  On both sides
of these lines the instance lists must be the ones the projected arrays call for: ordered by (tile, depth key, index),
every Gaussian as often as it touches tiles, with the ranges and the depth order that go with them."""
import numpy as np
import pytest

from paper_2609_05255_b200 import scenes
from gpu_helpers import run_gpu

pytestmark = pytest.mark.gpu


def _check(sc, cam):
    gpu = run_gpu(sc, cam)
    if gpu.P == 0:                                                       # nothing is ordered then
        assert not gpu.tile_ranges.any()
        return gpu
    visible = np.flatnonzero(gpu.visible)
    order = visible[np.lexsort((visible, gpu.depth_key[visible]))]
    assert np.array_equal(gpu.depth_order[:order.size], order)
    rest = np.setdiff1d(np.arange(gpu.n), visible)
    assert np.array_equal(gpu.depth_order[order.size:], rest)            # culled Gaussians, by index
    tiles, vals = gpu.sorted_tiles.astype(np.int64), gpu.sorted_vals.astype(np.int64)
    rank = np.empty(gpu.n, np.int64)
    rank[gpu.depth_order.astype(np.int64)] = np.arange(gpu.n)
    assert np.all(np.diff(tiles * gpu.n + rank[vals]) > 0)               # (tile, depth, index) ascending, no pair twice
    assert np.array_equal(np.bincount(vals, minlength=gpu.n), gpu.tiles_touched)
    gx = (cam.width + 15) // 16
    r = gpu.rect[vals]
    assert np.all((tiles % gx >= r[:, 0]) & (tiles % gx < r[:, 2]) & (tiles // gx >= r[:, 1]) & (tiles // gx < r[:, 3]))
    ranges = gpu.tile_ranges.reshape(-1, 2).astype(np.int64)
    counts = np.bincount(tiles, minlength=len(ranges))
    assert np.array_equal(ranges[:, 1] - ranges[:, 0], counts)
    assert np.array_equal(ranges[counts > 0, 0], (np.cumsum(counts) - counts)[counts > 0])
    return gpu


@pytest.mark.parametrize("n", [1, 2, 33, 1025, 2047, 2048, 2049, 5000, 8191, 8192, 8193, 16385, 32769])
def test_scene_sizes(n):
    sc = scenes.box_scene(n, 3.0, -1.0, 8.0, -3.5, 0.8, 1.0, scenes.APP_NEURAL, seed=500 + n)      # some behind the camera
    _check(sc, scenes.identity_camera(333, 217, 300.0))


@pytest.mark.parametrize("width,height", [(1, 1), (64, 64), (65, 1), (2048, 1024), (2049, 1025)])    # 1, 1, 2, 512, 561 cells
def test_image_sizes_and_large_footprints(width, height):
    sc = scenes.box_scene(3000, 3.0, 2.0, 8.0, -2.0, 1.0, 1.0, scenes.APP_SH, seed=9)
    gpu = _check(sc, scenes.identity_camera(width, height, float(max(width, height))))
    if width >= 2048:
        spans = (gpu.rect[:, 2] - 1) // 4 - gpu.rect[:, 0] // 4
        assert np.any(spans[gpu.visible] > 2)                            # footprints of more than 3 x 3 cells


@pytest.mark.parametrize("n", [1, 33, 1025, 8192])
def test_few_gaussians_through_the_grid_wide_kernels(n):
    """561 cells are too many for the cluster: the way that small scenes take where a cluster cannot be launched."""
    sc = scenes.box_scene(n, 3.0, -1.0, 8.0, -3.5, 0.8, 1.0, scenes.APP_NEURAL, seed=600 + n)
    _check(sc, scenes.identity_camera(2049, 1025, 1500.0))


@pytest.mark.parametrize("n", [1500, 8000, 20011])
def test_equal_depths_keep_the_index_order(n):
    sc = scenes.box_scene(n, 2.0, 3.0, 3.0, -3.0, 0.5, 1.0, scenes.APP_SH, seed=3)
    assert np.all(sc.means[:, 2] == 3.0)
    _check(sc, scenes.identity_camera(256, 200, 256.0))


def test_nothing_visible():
    sc = scenes.box_scene(5000, 2.0, -8.0, -3.0, -3.0, 0.5, 1.0, scenes.APP_SH, seed=4)
    gpu = run_gpu(sc, scenes.identity_camera(128, 96, 128.0), pair_capacity=64)
    assert gpu.P == 0 and not gpu.tile_ranges.any()
