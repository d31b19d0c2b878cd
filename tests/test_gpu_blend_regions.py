"""The blend kernels give every warp a region of a tile and choose its size by the number of tiles (backward: 4 x 8 pixels
up to 64 tiles, and up to 100 with 50 Gaussians per tile, 8 x 8 up to 1000, up to 3200 with 50 and up to 6000 with 350, 16 x 8
beyond); lists go through shared memory 32 entries at a time, in groups of four, and what the lanes park is summed every eight
entries.  Checked against the oracle at the edges of all of these: tile counts and scene sizes on either side of every line,
ragged images, lists of about 32 and 64 entries, opacities above the alpha clamp."""
import copy

import numpy as np
import pytest

from paper_2609_05255_b200 import scenes
from gpu_helpers import grad_mismatch, grad_names, image_mismatch, run_gpu

pytestmark = pytest.mark.gpu


LINES = [(3_000, 640, 400), (3_000, 1025, 247),                                  # 1000, 1040 tiles
         (159_999, 800, 1024), (160_000, 800, 1024), (170_000, 1617, 512),       # 3200 tiles and 50 per tile; 3264
         (2_099_999, 960, 1600), (2_100_000, 960, 1600), (2_200_000, 961, 1600)] # 6000 tiles and 350 per tile; 6100


def _check(oracle, sc, cam, allow=0.01):   # sums over 800 x 950 pixels, of both signs: 0.3 % miss the literal rule
    G = scenes.upstream_gradient(cam, 5)
    gpu = run_gpu(sc, cam, G)
    fwd, ref = oracle.render(sc, cam, G)
    assert not image_mismatch(gpu.image, fwd.image, fwd.fragile).any()
    differ = gpu.n_contrib != fwd.n_contrib.reshape(gpu.n_contrib.shape)
    assert not differ[~fwd.fragile.astype(bool)].any()
    for nm in grad_names(sc.app):
        bad = grad_mismatch(getattr(gpu.grads, nm), getattr(ref, nm))
        assert bad.mean() <= allow, (nm, int(bad.sum()))


@pytest.mark.parametrize("width,height", [(1, 1), (9, 17), (128, 128), (130, 127), (800, 952), (803, 953)])
def test_image_sizes_at_the_lines_between_region_sizes(oracle, width, height):
    sc = scenes.box_scene(3000, 2.0, 2.0, 6.0, -3.0, 0.5, 1.0, scenes.APP_SH, seed=31)
    cam = scenes.identity_camera(width, height, float(max(width, height)), background=(0.2, 0.1, 0.3))
    _check(oracle, sc, cam)


@pytest.mark.parametrize("width,height", [(160, 160), (1601, 16), (640, 400), (1025, 247), (800, 1280), (1022, 1008)])
def test_on_either_side_of_the_lines(oracle, width, height):
    """100 and 101 tiles (both 8 x 8 pixels for so few Gaussians), 1000 and 1040 (8 x 8, 16 x 8), 4000 and 4032 (16 x 8)."""
    sc = scenes.box_scene(3000, 2.0, 2.0, 6.0, -3.0, 0.5, 1.0, scenes.APP_SH, seed=32)
    _check(oracle, sc, scenes.identity_camera(width, height, float(max(width, height)), background=(0.2, 0.1, 0.3)))


def _few_and_many(n):
    few = scenes.box_scene(3000, 2.0, 2.0, 6.0, -3.0, 0.5, 1.0, scenes.APP_NEURAL, seed=33)
    many = copy.copy(few)
    for name in ("means", "log_scales", "quats", "opacity_logits", "base_color", "features"):
        a = getattr(few, name)
        setattr(many, name, np.concatenate([a, np.repeat(a[:1], n - 3000, 0)]))
    many.means[3000:, 2] = -3.0
    return few, many


@pytest.mark.parametrize("n,width,height", [(4_999, 160, 160), (5_000, 160, 160),                  # 100 tiles: 8 x 8 pixels, 4 x 8
                                            (1_203_199, 1021, 752), (1_203_200, 1021, 752)])       # 3008 tiles: 8 x 8
def test_many_gaussians_for_their_tiles(oracle, n, width, height):
    """3000 Gaussians in view, the others behind the camera: the size of the scene alone chooses the kernel."""
    few, many = _few_and_many(n)
    cam = scenes.identity_camera(width, height, float(width))
    G = scenes.upstream_gradient(cam, 5)
    gpu = run_gpu(many, cam, G)
    fwd, ref = oracle.render(few, cam, G)
    assert image_mismatch(gpu.image, fwd.image, fwd.fragile).mean() <= 1e-4
    for nm in grad_names(few.app):
        got = getattr(gpu.grads, nm)
        if nm != "mlp_weights":
            assert not got[3000:].any(), nm
            got = got[:3000]
        bad = grad_mismatch(got, getattr(ref, nm))
        assert bad.mean() <= 0.01, (nm, int(bad.sum()))


@pytest.mark.parametrize("n,width,height", LINES)
def test_the_lines_for_larger_images(oracle, n, width, height):
    test_many_gaussians_for_their_tiles(oracle, n, width, height)


@pytest.mark.parametrize("n,width,height", LINES)
def test_every_pixel_at_the_lines_for_larger_images(oracle, n, width, height):
    few, many = _few_and_many(n)
    cam = scenes.identity_camera(width, height, float(width))
    gpu = run_gpu(many, cam, scenes.upstream_gradient(cam, 5))
    fwd, _ = oracle.render(few, cam)
    assert not image_mismatch(gpu.image, fwd.image, fwd.fragile).any()
    # n_contrib is a place in the tile's list: compared where both sides list the same number (a footprint that ends within rounding of a
    # tile's first pixels may be listed on one side only: 3000 of them with edges good to 1e-4 of a pixel, one or two tiles here)
    lists = gpu.tile_ranges.reshape(-1, 2).astype(np.int64)
    same = (lists[:, 1] - lists[:, 0] == fwd.ranges[:, 1].astype(np.int64) - fwd.ranges[:, 0]).reshape((height + 15) // 16, (width + 15) // 16)
    assert (~same).sum() <= 4
    pixels = np.repeat(np.repeat(same, 16, 0), 16, 1)[:height, :width] & ~fwd.fragile.astype(bool)
    assert np.array_equal(gpu.n_contrib[pixels], fwd.n_contrib.reshape(gpu.n_contrib.shape)[pixels])


@pytest.mark.parametrize("n", [1, 3, 4, 5, 7, 8, 9, 31, 32, 33, 40, 63, 64, 65])
def test_list_lengths_around_the_pieces(oracle, n):
    # every Gaussian covers the one tile of the image with a low opacity: the whole list is composited
    sc = scenes.box_scene(n, 0.05, 2.0, 4.0, -1.0, 0.1, 0.1, scenes.APP_NEURAL, seed=40 + n)
    sc.opacity_logits[:] = -4.0
    _check(oracle, sc, scenes.identity_camera(16, 13, 16.0))


def test_opacities_above_the_clamp(oracle):
    sc = scenes.box_scene(2000, 1.0, 2.0, 4.0, -2.0, 0.5, 1.0, scenes.APP_SH, seed=77)
    sc.opacity_logits[::3] = 7.0
    _check(oracle, sc, scenes.identity_camera(96, 80, 96.0))
