"""The instance count of a view is taken by the warps of the preprocess, each over a run of Gaussians, and summed in one word
beside the number of warps.  It must be exact however large it gets: more than 2^32 instances in the run of one warp, more
than 2^40 in the view (the largest count that the report to the host holds), and the views after such a one must count
right too."""
import pytest

from paper_2609_05255_b200 import scenes

pytestmark = pytest.mark.gpu


def _covering(api, torch, n):
    """n equal Gaussians, each on every tile of the largest image; degree 0, so that nothing is decoded."""
    f = dict(device="cuda", dtype=torch.float32)
    means = torch.tensor([0.0, 0.0, 4.0], **f).repeat(n, 1)
    zeros = torch.zeros((n, 3), **f)
    quats = torch.tensor([1.0, 0.0, 0.0, 0.0], **f).repeat(n, 1)
    return api.DeviceScene(means, zeros + 3.0, quats, zeros[:, 0] + 2.0, base_color=zeros, app=scenes.APP_NEURAL, active_degree=0,
                           features=torch.zeros((n, 8), device="cuda", dtype=torch.float16),
                           mlp_weights=torch.zeros((api.MLP_WEIGHTS,), device="cuda", dtype=torch.float16))


def test_counts_beyond_32_and_40_bits():
    import torch
    from paper_2609_05255_b200 import api
    ctx = api.Context(0)
    cam = api.make_camera(scenes.identity_camera(16384, 16384, 16384.0))
    small = _covering(api, torch, 3)
    small_proj = api.alloc_projected(3, ctx.device, False)
    each = api.gs_preprocess(ctx, small, cam, small_proj) // 3
    assert each == 1 << 20
    count = 16_000_000                               # on 3552 warps (of 888 CTAs) 4505 Gaussians each: 2^32.1 instances a warp
    scene, proj = _covering(api, torch, count), api.alloc_projected(count, ctx.device, False)
    assert api.gs_preprocess(ctx, scene, cam, proj) == count * each
    # the device-counted path: the count of the large view, the lists of a small one
    view = scenes.identity_camera(64, 64, 64.0)
    r = api.Renderer(ctx, 3, 64, 64, small.app, pair_capacity=64)
    api.gs_preprocess(ctx, small, api.make_camera(view), r.proj)
    api.gs_preprocess_async(ctx, scene, cam, proj)
    api.gs_render_forward(ctx, 3, r.proj, api.make_camera(view), api.GS_PAIRS_ON_DEVICE, 64, r.binning, r.image, r.final_T, r.n_contrib,
                          r.workspace)
    assert api.gs_async_pairs(ctx) == count * each
    with pytest.raises(api.GsError):
        api.gs_async_status(ctx)                     # more than the capacity
    # and the next view counts from zero again
    assert api.gs_preprocess(ctx, small, cam, small_proj) == 3 * each
    r.forward(small, api.make_camera(view))
    assert r.num_pairs == 3 * 16
    ctx.close()
