"""The path without host waits: gs_preprocess_async + gs_render_forward(GS_PAIRS_ON_DEVICE) must give the
same bits as the path that reads the instance count back, and an overflow of the capacity must be
reported (with every write kept inside the caller's buffers)."""
import numpy as np
import pytest

from paper_2609_05255_b200 import scenes

pytestmark = pytest.mark.gpu


def _setup(n=20_011, app=scenes.APP_NEURAL):
    import torch
    from paper_2609_05255_b200 import api
    w = scenes.config2(n=n, app=app)
    ctx = api.Context(0)
    ds = api.upload_scene(w.scene, ctx.device)
    cam = api.make_camera(w.cameras[0])
    return torch, api, ctx, ds, cam, w


def test_device_counted_view_equals_host_counted_view():
    torch, api, ctx, ds, cam, w = _setup()
    W, H = w.cameras[0].width, w.cameras[0].height
    probe = api.alloc_projected(ds.n, ctx.device, False)
    P = api.gs_preprocess(ctx, ds, cam, probe)
    cap = int(P * 1.3) + 777
    a = api.Renderer(ctx, ds.n, W, H, ds.app, pair_capacity=cap)
    b = api.Renderer(ctx, ds.n, W, H, ds.app, pair_capacity=cap)
    G = torch.from_numpy(scenes.upstream_gradient(w.cameras[0], 5)).to(ctx.device)
    a.forward(ds, cam); a.backward(ds, cam, G)
    b.forward_async(ds, cam); b.backward(ds, cam, G)
    api.gs_async_status(ctx)
    assert torch.equal(a.image, b.image) and torch.equal(a.final_T, b.final_T) and torch.equal(a.n_contrib, b.n_contrib)
    assert torch.equal(a.binning.tile_ranges, b.binning.tile_ranges)
    assert torch.equal(a.binning.sorted_vals[:P], b.binning.sorted_vals[:P])
    for k in ("means", "log_scales", "quats", "opacity_logits", "base_color", "features"):
        x, y = getattr(a.grads, k), getattr(b.grads, k)
        # the blend backward sums with atomics: equal up to the order of those sums.  Two runs of the SAME path differ
        # by up to 3e-7 of the largest gradient of the kind (measured: 2.3e-5 on gradients of up to 87)
        assert (x - y).abs().max().item() <= 2e-6 * x.abs().max().item(), k
    ctx.close()


def test_overflow_is_reported_and_nothing_is_written_past_the_capacity():
    torch, api, ctx, ds, cam, w = _setup()
    W, H = w.cameras[0].width, w.cameras[0].height
    probe = api.alloc_projected(ds.n, ctx.device, False)
    P = api.gs_preprocess(ctx, ds, cam, probe)
    cap = P // 3
    r = api.Renderer(ctx, ds.n, W, H, ds.app, pair_capacity=cap)
    # canaries behind the instance lists (the buffers hold exactly `cap` entries, allocated apart)
    guard = 4096
    big_t = torch.full((cap + guard,), 0x5A5A5A5A, device=ctx.device, dtype=torch.int32)
    big_v = torch.full((cap + guard,), 0x5A5A5A5A, device=ctx.device, dtype=torch.int32)
    r.binning.sorted_tiles, r.binning.sorted_vals = big_t[:cap], big_v[:cap]
    r.forward_async(ds, cam)
    with pytest.raises(api.GsError) as e:
        api.gs_async_status(ctx)
    assert e.value.status == api.GS_ERR_CAPACITY
    assert torch.all(big_t[cap:] == 0x5A5A5A5A) and torch.all(big_v[cap:] == 0x5A5A5A5A)
    api.gs_async_status(ctx)                      # the flag was cleared
    # the same renderer with the host-counted call refuses up front
    with pytest.raises(api.GsError) as e:
        r.forward(ds, cam)
    assert e.value.status == api.GS_ERR_CAPACITY
    ctx.close()


def test_empty_scene_through_the_async_calls():
    import torch
    from paper_2609_05255_b200 import api
    ctx = api.Context(0)
    sc = scenes.config1(0).scene if hasattr(scenes, "config1") else None
    ds = api.upload_scene(sc, ctx.device)
    cam_h = scenes.identity_camera(64, 64, 64.0)
    cam = api.make_camera(cam_h)
    r = api.Renderer(ctx, 0, 64, 64, ds.app, pair_capacity=16)
    r.forward_async(ds, cam)
    api.gs_async_status(ctx)
    bg = torch.tensor(np.asarray(cam_h.background, np.float32), device=ctx.device)
    assert torch.equal(r.image, bg[:, None, None].expand(3, 64, 64))
    ctx.close()


def _pairs_of_views(api, ctx, ds, cam):
    probe = api.alloc_projected(ds.n, ctx.device, False)
    return api.gs_preprocess(ctx, ds, cam, probe)


def test_pairs_of_a_replayed_graph_are_those_of_the_replay():
    torch, api, ctx, ds, cam, w = _setup()
    W, H = w.cameras[0].width, w.cameras[0].height
    other = api.Context(0)
    before = _pairs_of_views(api, other, ds, cam)
    r = api.Renderer(ctx, ds.n, W, H, ds.app, pair_capacity=int(before * 1.3) + 777)
    r.forward(ds, cam)
    assert r.num_pairs == before
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        r.forward_async(ds, cam, stream=stream)
        with pytest.raises(api.GsError) as e:
            api.gs_async_pairs(ctx, stream=stream)               # refused, and the capture stays whole
        assert e.value.status == api.GS_ERR_INVALID_ARG
    with torch.cuda.stream(stream):
        graph.replay()
        assert api.gs_async_pairs(ctx) == before
        ds.means[: ds.n // 2] = 1e3                              # half of the scene leaves the view
        after = _pairs_of_views(api, other, ds, cam)
        assert 0 < after < before
        torch.cuda._sleep(20_000_000)                            # the replay is still to come when the count is asked for
        graph.replay()
        assert api.gs_async_pairs(ctx) == after
    # a view issued by a call answers for itself again
    torch.cuda.synchronize()
    r.forward(ds, cam)
    assert r.num_pairs == after
    del graph
    ctx.close(); other.close()


def test_a_capacity_of_zero_overflows_like_any_other():
    torch, api, ctx, ds, cam, w = _setup(n=5_003)
    W, H = w.cameras[0].width, w.cameras[0].height
    P = _pairs_of_views(api, ctx, ds, cam)
    full = api.Renderer(ctx, ds.n, W, H, ds.app, pair_capacity=P)
    none = api.Renderer(ctx, ds.n, W, H, ds.app, pair_capacity=0)
    full.forward_async(ds, cam)
    assert api.gs_async_pairs(ctx) == P
    api.gs_async_status(ctx)                                     # within the capacity
    assert api.gs_async_pairs(ctx) == P                          # asked again, after the stream has drained
    none.forward_async(ds, cam)
    assert api.gs_async_pairs(ctx) == P
    with pytest.raises(api.GsError) as e:
        api.gs_async_status(ctx)
    assert e.value.status == api.GS_ERR_CAPACITY
    empty = api.upload_scene(scenes.config1(0).scene, ctx.device)
    e = api.Renderer(ctx, 0, 64, 64, empty.app, pair_capacity=0)
    e.forward_async(empty, api.make_camera(scenes.identity_camera(64, 64, 64.0)))
    assert api.gs_async_pairs(ctx) == 0
    api.gs_async_status(ctx)
    ctx.close()
