"""Per-Gaussian backward of the explicit models (SH, Spherical Voronoi).  A CTA takes 128 words of 32 Gaussians at a time: words
in which at least 20 received a gradient move whole, the Gaussians of the others are listed and gathered.  Checked against
the oracle with words of every filling, ragged ends and a degree without rows; a Gaussian without a gradient must keep exact
zeros, and whatever its parameters are must not reach its neighbours in a word that moves whole; scenes so large that a
CTA has more than one round must agree with the same Gaussians alone."""
import copy

import numpy as np
import pytest

from paper_2609_05255_b200 import scenes
from gpu_helpers import grad_mismatch, grad_names, run_gpu

pytestmark = pytest.mark.gpu

ROWS = {scenes.APP_SH: "sh_rest", scenes.APP_SV: "sv_sites"}


def _scene(app, n, keep, seed):
    """A box of faint Gaussians, so that all that are in view receive a gradient; those outside `keep` lie behind the camera."""
    sc = scenes.box_scene(n, 0.7, 2.0, 4.0, -3.5, 0.3, 0.1, app, seed=seed)
    sc.opacity_logits[:] = -3.0
    sc.means[~keep, 2] = -3.0
    return sc


@pytest.mark.parametrize("degree", [3, 1, 0])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 19 * 32 + 20, 33 * 32, 200 * 32 + 7])
@pytest.mark.parametrize("app", [scenes.APP_SH, scenes.APP_SV], ids=["sh", "sv"])
def test_words_of_every_filling(oracle, app, n, degree):
    i = np.arange(n)
    keep = (i * 7) % 32 < (i // 32 * 5 + 20) % 33              # 20, 25, 30, 2, ... of the 32 Gaussians of a word
    sc = _scene(app, n, keep, 70 + n)
    sc.active_degree = degree
    cam = scenes.identity_camera(100, 90, 100.0)
    G = scenes.upstream_gradient(cam, 5)
    _, ref = oracle.render(sc, cam, G)
    sick = copy.copy(sc)
    rows = getattr(sc, ROWS[app]).copy()
    rows[~keep] = np.nan
    setattr(sick, ROWS[app], rows)
    gpu = run_gpu(sick, cam, G)
    assert np.array_equal((gpu.g2d[:, :9] != 0).any(1), keep)
    for nm in grad_names(app):
        got, want = getattr(gpu.grads, nm), getattr(ref, nm)
        assert np.all(np.asarray(got)[~keep] == 0), nm
        bad = grad_mismatch(got, want)
        assert bad.mean() <= 0.002, (nm, int(bad.sum()))


@pytest.mark.parametrize("app", [scenes.APP_SH, scenes.APP_SV], ids=["sh", "sv"])
def test_more_than_one_round(app):
    """4.2M Gaussians are 177 words for each of 740 CTAs; nearly all lie behind the camera."""
    import torch
    from paper_2609_05255_b200 import api
    n, view = 4_200_011, scenes.identity_camera(200, 160, 200.0)
    keep = torch.zeros(n, dtype=torch.bool, device="cuda")
    keep[::1500] = True                                       # thin words, in every round
    for first in (1_000_000, 2_718_720, n - 1500):            # and full ones, the last of them ragged
        keep[first:first + 1500] = True
    ids = keep.nonzero().squeeze(1)
    small = _scene(app, len(ids), np.ones(len(ids), bool), 11)
    ctx, cam = api.Context(0), api.make_camera(view)
    G = torch.from_numpy(scenes.upstream_gradient(view, 5)).to(ctx.device)

    def gradients(ds):
        probe = api.alloc_projected(ds.n, ctx.device, False)
        r = api.Renderer(ctx, ds.n, view.width, view.height, app, pair_capacity=api.gs_preprocess(ctx, ds, cam, probe))
        r.forward(ds, cam)
        return r.backward(ds, cam, G)

    one = api.upload_scene(small, ctx.device)
    want = gradients(one)
    names = ["means", "log_scales", "quats", "opacity_logits", "base_color", ROWS[app]]
    behind = {"means": -3.0}
    big = {nm: torch.full((n,) + getattr(one, nm).shape[1:], behind.get(nm, 0.25), device=ctx.device) for nm in names}
    for nm in names:
        big[nm][ids] = getattr(one, nm)
    got = gradients(api.DeviceScene(*[big[nm] for nm in names[:5]], app=app, active_degree=3, **{ROWS[app]: big[names[5]]}))
    for nm in names:
        g, w = getattr(got, nm), getattr(want, nm)
        assert not bool((g[~keep] != 0).any()), nm
        # the same sums over pixels in another order (the launch differs in nothing else): 2e-6 of the largest in
        # test_gpu_async; through the inverse covariance of these round Gaussians a few times that
        assert float((g[ids] - w).abs().max()) <= 2e-5 * float(w.abs().max()), nm
    ctx.close()
