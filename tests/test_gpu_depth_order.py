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
@pytest.mark.parametrize("n,z_lo", [(32769, 2.0), (40001, -6.0), (33000, -300.0), (151552, -6.0), (151553, -6.0)])  # none, half, nearly all culled; blocks of 512 and 1024
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


def _hidden(n):
    """Where the sample of the keys is taken."""
    stride = min(2048, max(256, n // 148)) // 8
    j = np.arange((n + stride - 1) // stride, dtype=np.uint64)
    at = j * np.uint64(stride) + ((j * np.uint64(2654435761) & np.uint64(0xffffffff)) * np.uint64(stride) >> np.uint64(32))
    return at[at < n].astype(np.int64)


@pytest.mark.parametrize("kind", ["nested", "three_large", "grid", "many_planes", "large_planes"])
@pytest.mark.parametrize("n", [12_000, 60_001, 600_000])
def test_bins_that_are_split_again(kind, n):
    rng = np.random.default_rng(n + 1)
    if kind == "nested":                       # a few, a few close to the others, and the others at one depth: what a second split leaves crowded
        depths = np.full(n, 4.0, np.float32)
        depths[rng.permutation(n)[:20]] = np.concatenate([rng.uniform(2.0, 2.1, 4), rng.uniform(3.999, 3.9995, 8),
                                                          rng.uniform(4.0005, 4.001, 5), rng.uniform(7.0, 8.0, 3)])
    elif kind == "three_large":                # two splitters, and three buckets beyond shared memory from 60 001 on
        depths = rng.uniform(2.0, 8.0, n)
        at = _hidden(n)
        depths[at] = -5.0
        depths[at[:16]] = np.repeat([4.0, 6.0], 8)
    elif kind == "large_planes":               # the same in four planes
        depths = rng.choice([2.5, 3.0, 6.0, 7.0], n)
        depths[_hidden(n)] = -5.0
    elif kind == "grid":                       # as many planes as rows and columns, neighbours in memory in different ones
        depths = 2.0 + 6.0 * (np.arange(n) % round(n ** (1 / 3))) / round(n ** (1 / 3))
    else:                                      # several planes to a bucket
        depths = 2.0 + 6.0 * rng.integers(0, n // 300, n) / (n // 300)
    gpu = _check(_scene_at(np.float32(depths), n), scenes.identity_camera(333, 217, 300.0))
    if kind in ("three_large", "large_planes") and n > 12_000:
        assert gpu.visible.sum() > 3 * 7680


def test_nearly_all_of_the_largest_scene_in_one_bucket():
    """The parts of the bucket hold more than a CTA keeps, and are taken in turns."""
    n = 4_194_304
    sc = scenes.box_scene(n, 3.0, 2.0, 8.0, -6.0, 0.5, 1.0, scenes.APP_NEURAL, seed=8)
    sc.means[_hidden(n), 2] = -5.0
    assert _check(sc, scenes.identity_camera(333, 217, 300.0)).visible.sum() > 2_000_000


def _time_of_ordering(depths):
    """Microseconds of the depth order, median of several forwards."""
    import torch
    from paper_2609_05255_b200 import api
    n, (width, height) = len(depths), (400, 400)
    ctx = api.Context(0)
    gen = torch.Generator(device=ctx.device)
    gen.manual_seed(3)
    z = torch.from_numpy(np.float32(depths)).to(ctx.device)
    xy = (torch.rand((n, 2), device=ctx.device, generator=gen) - 0.5) * z.abs()[:, None]
    sizes = torch.log(z.abs() / 400.0)[:, None].expand(n, 3).contiguous()
    zeros = torch.zeros((n, 8), device=ctx.device)
    sc = api.DeviceScene(torch.cat([xy, z[:, None]], 1).contiguous(), sizes, torch.ones((n, 4), device=ctx.device), zeros[:, 0].contiguous(),
                         app=api.GS_APP_NEURAL, active_degree=0, base_color=zeros[:, :3].contiguous(), features=zeros.half(),
                         mlp_weights=torch.zeros(816, device=ctx.device).half())
    cam = api.make_camera(scenes.identity_camera(width, height, 400.0))
    pairs = api.gs_preprocess(ctx, sc, cam, api.alloc_projected(n, ctx.device))
    r = api.Renderer(ctx, n, width, height, sc.app, pairs)
    times = []
    for _ in range(12):
        api.gs_profile_enable(ctx, True)
        r.forward(sc, cam)
        torch.cuda.synchronize()
        times.append(api.gs_profile_collect(ctx)[0]["depth_sort"] * 1e3)
    ctx.close()
    return float(np.median(times[3:]))


def test_time_does_not_depend_on_the_depths():
    """1M Gaussians: measured 1.5 times as long as evenly spread depths at most (2.6 to 3 times where crowded bins were sorted by
    comparators, 60 times with one bucket of 65 536 in memory)."""
    n, rng = 1_000_000, np.random.default_rng(1)
    even = _time_of_ordering(rng.uniform(2.0, 8.0, n))
    outliers = np.where(rng.random(n) < 0.95, rng.uniform(4.0, 4.1, n), np.exp(rng.uniform(np.log(0.3), np.log(300.0), n)))
    hidden = rng.uniform(2.0, 8.0, n)
    hidden[_hidden(n)] = -5.0
    hidden[65_536:] = -5.0
    for name, depths in (("outliers", outliers), ("1000 planes", 2.0 + rng.integers(0, 1000, n) * 0.006),
                         ("20000 planes", 2.0 + rng.integers(0, 20_000, n) * 0.0003), ("one bucket", hidden)):
        t = _time_of_ordering(depths)
        assert t <= 2.2 * even, (name, t, even)
