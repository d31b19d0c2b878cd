"""The gradient rows of Gaussians that receive nothing are written by the warps of the blend backward, each a slice of all
rows.  An image of few tiles gets further warps for it.  Whatever the image, every row must be written: the buffers start
as NaN, and afterwards all is finite, zero where the 2D gradients are zero and only there (the upstream gradient is dense)."""
import pytest

from paper_2609_05255_b200 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,height", [(1, 1), (16, 16), (70, 40), (320, 200)])       # 8, 8, 120 (8 x 15), 1040 warps with a region
@pytest.mark.parametrize("n", [1, 3, 999, 60_001])                                       # 60 001: more than two warps per SM at 4 KB each
@pytest.mark.parametrize("app", [scenes.APP_SH, scenes.APP_NEURAL, scenes.APP_SV], ids=["sh", "neural", "sv"])
def test_every_row_is_written(app, n, width, height):
    import torch
    from paper_2609_05255_b200 import api
    ctx = api.Context(0)
    w = scenes.config3(app, n=n, width=width, height=height, views=1) if n > 1000 else None
    sc = w.scene if w else scenes.box_scene(n, 1.0, 2.0, 4.0, -3.0, 0.5, 1.0, app, seed=n)
    cam_h = w.cameras[0] if w else scenes.identity_camera(width, height, float(max(width, height)))
    ds, cam = api.upload_scene(sc, ctx.device), api.make_camera(cam_h)
    probe = api.alloc_projected(n, ctx.device, False)
    r = api.Renderer(ctx, n, width, height, app, pair_capacity=max(api.gs_preprocess(ctx, ds, cam, probe), 1))
    names = ["means", "log_scales", "quats", "opacity_logits", "base_color"] + {
        scenes.APP_SH: ["sh_rest"], scenes.APP_NEURAL: ["features"], scenes.APP_SV: ["sv_sites"]}[app]
    for nm in names:
        getattr(r.grads, nm).fill_(float("nan"))
    r.forward(ds, cam)
    r.backward(ds, cam, torch.from_numpy(scenes.upstream_gradient(cam_h, 5)).to(ctx.device))
    torch.cuda.synchronize()
    none = ~(r.workspace[: n * 48].view(torch.float32).reshape(n, 12)[:, :9] != 0).any(1)
    for nm in names:
        rows = getattr(r.grads, nm).reshape(max(n, 1), -1)[:n]
        assert bool(torch.isfinite(rows).all()), nm
        assert not bool((rows[none] != 0).any()), nm
    assert n <= 1000 or bool(none.any())
    if bool((~none).any()):
        assert bool((r.grads.base_color[:n][~none] != 0).any())
    ctx.close()
