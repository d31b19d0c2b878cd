"""Images of up to 65535 tile rows, the most that a camera may have: Gaussians above and below tile row 32768 (and close to the last
row) must be listed in the tiles that they meet, be composited and receive their gradients.  Projected centres of that size are
only good to 1/32 of a pixel in single precision, so everything is compared with the oracle on the projected values themselves."""
import dataclasses

import numpy as np
import pytest

from paper_2609_05255_b200 import scenes
from gpu_helpers import grad_mismatch, image_mismatch, run_gpu

pytestmark = pytest.mark.gpu

DEPTH = 4.0


def _column(app, width, height, rows, per_row, pixels, seed):
    """`per_row` Gaussians about each of the tile rows, of about `pixels` standard deviation."""
    rng = np.random.default_rng(seed)
    cam = dataclasses.replace(scenes.identity_camera(width, height, height / 2.0), fx=64.0)
    n = len(rows) * per_row
    sc = scenes.box_scene(n, 1.0, DEPTH, DEPTH, 0.0, 0.0, 1.0, app, seed=seed)
    y = (np.repeat(rows, per_row) + rng.uniform(0.0, 1.0, n)) * 16.0
    x = rng.uniform(0.0, width, n)
    means = np.stack([(x - cam.cx) / cam.fx * DEPTH, (y - cam.cy) / cam.fy * DEPTH, np.full(n, DEPTH)], 1)
    scale = np.stack([np.full(n, pixels * DEPTH / cam.fx), np.full(n, pixels * DEPTH / cam.fy), np.full(n, 1e-9)], 1)
    quats = np.tile(np.float32([1, 0, 0, 0]), (n, 1))
    return dataclasses.replace(sc, means=means.astype(np.float32), log_scales=np.log(scale).astype(np.float32), quats=quats), cam


@pytest.mark.parametrize("app", [scenes.APP_SH, scenes.APP_NEURAL, scenes.APP_SV])
@pytest.mark.parametrize("width,tile_rows,pixels", [(16, 33_000, 3.0), (24, 40_000, 1.0), (16, 65_535, 3.0), (16, 65_535, 40.0)])  # 40: large footprints
def test_tile_rows_beyond_32768(oracle, app, width, tile_rows, pixels):
    height = 16 * tile_rows
    rows = np.array([2, 100, 32_700, 32_766, 32_767, 32_768, 32_769, 32_900, tile_rows - 200, tile_rows - 3])
    sc, cam = _column(app, width, height, rows, 24, pixels, tile_rows + width)
    G = np.zeros((3, height, width), np.float32)
    for r in rows:                                                    # upstream gradients where there is something to see
        lo, hi = max(16 * (r - 8), 0), min(16 * (r + 9), height)
        G[:, lo:hi] = np.random.default_rng(r).normal(size=(3, hi - lo, width))
    gpu = run_gpu(sc, cam, G)
    rect, tiles, pairs = oracle.tile_spans_f32(gpu.extent[:, 0] >= 0, gpu.mean2d, gpu.chol, gpu.extent, width, height)
    assert np.array_equal(gpu.rect, rect) and np.array_equal(gpu.tiles_touched, tiles) and gpu.P == pairs
    row = np.floor(gpu.mean2d[:, 1] / 16)
    assert gpu.visible.mean() > 0.9 and gpu.visible[row >= 32_768].mean() > 0.9 and gpu.visible[row < 32_768].mean() > 0.9
    keys, vals, ranges = oracle.sorted_instances_f32(rect, tiles, gpu.mean2d, gpu.chol, gpu.extent, np.where(gpu.visible, gpu.depth_key, 0), width, height, pairs)
    assert np.array_equal(gpu.sorted_vals, vals) and np.array_equal(gpu.tile_ranges.reshape(-1, 2), ranges)
    conic, opacity = gpu.conic_opacity[:, :3], gpu.conic_opacity[:, 3]
    want = oracle.blend_forward(cam, vals, ranges, gpu.mean2d, conic, opacity, gpu.color)
    assert not image_mismatch(gpu.image, want.image, want.fragile).any()
    g2 = oracle.blend_backward(cam, vals, ranges, gpu.mean2d, conic, opacity, gpu.color, G, with_abs=True)
    # an fp32 sum of terms of both signs, and whole terms where a pair lies within rounding of a blend threshold
    allowed = g2.abs_sum[:, :3] + 1.5 * g2.flip_sum[:, :3] / 1e-5
    assert not grad_mismatch(gpu.grads.base_color, np.where(gpu.color > 0, g2.color, 0.0), allowed).any()
    reached = gpu.grads.means.any(1)
    assert reached[gpu.visible].mean() > 0.8 and reached[(row >= 32_768) & gpu.visible].mean() > 0.8
