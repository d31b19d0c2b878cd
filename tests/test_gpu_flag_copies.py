"""The flags of who received a gradient exist up to sixteen times for scenes of less than 65 536 Gaussians, a warp of the blend
backward setting those of one copy.  (With a tile for every 20 of them.)  A Gaussian that a single pixel composites is flagged in one copy only, whichever it
is, and must get its gradients: single lit pixels all over an image, at the scene sizes where the number of copies changes, in
all consumers of the flags."""
import numpy as np
import pytest

from paper_2609_05255_b200 import scenes
from gpu_helpers import grad_mismatch, grad_names, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 33, 4096, 8500, 8501])                               # 16 copies, and 1 at 8501: 425 tiles
@pytest.mark.parametrize("app", [scenes.APP_SH, scenes.APP_NEURAL, scenes.APP_SV], ids=["sh", "neural", "sv"])
def test_single_pixels(oracle, app, n):                                                # (25 x 17 tiles)
    sc = scenes.box_scene(n, 2.0, 2.0, 5.0, -4.5, 0.3, 1.0, app, seed=900 + n % 97)
    cam = scenes.identity_camera(400, 272, 260.0)
    G = np.zeros_like(scenes.upstream_gradient(cam, 5))
    G[:, 3::37, 5::41] = scenes.upstream_gradient(cam, 5)[:, 3::37, 5::41]                 # 8 x 10 pixels, a warp each
    gpu = run_gpu(sc, cam, G)
    _, ref = oracle.render(sc, cam, G)
    lit = (gpu.g2d[:, :9] != 0).any(1)
    assert n == 1 or (lit.any() and not lit.all())
    for nm in grad_names(app):
        got, want = np.asarray(getattr(gpu.grads, nm)), np.asarray(getattr(ref, nm))
        if nm != "mlp_weights":
            assert not np.any(got[~lit]), nm
        bad = grad_mismatch(got, want)
        assert bad.mean() <= 0.002, (nm, int(bad.sum()))
    if lit.any():
        assert np.all((gpu.grads.base_color[lit] != 0).any(1) | (gpu.color[lit] <= 0).any(1))


@pytest.mark.parametrize("n", [16_383, 16_384, 65_535, 65_536])                          # 16, 4, 4, 1 copies
def test_more_gaussians(oracle, n):
    sc = scenes.box_scene(n, 3.5, 2.0, 5.0, -5.0, 0.3, 1.0, scenes.APP_SH, seed=90)
    cam = scenes.identity_camera(1024, 816, 600.0)                                        # 64 x 51 tiles
    G = np.zeros_like(scenes.upstream_gradient(cam, 5))
    G[:, 3::97, 5::89] = scenes.upstream_gradient(cam, 5)[:, 3::97, 5::89]
    gpu = run_gpu(sc, cam, G)
    _, ref = oracle.render(sc, cam, G)
    for nm in grad_names(sc.app):
        bad = grad_mismatch(getattr(gpu.grads, nm), getattr(ref, nm))
        assert bad.mean() <= 0.002, (nm, int(bad.sum()))


def test_decoder_variant(oracle):
    n = 8_001
    sc = scenes.box_scene(n, 2.0, 2.0, 5.0, -4.5, 0.3, 1.0, scenes.APP_NEURAL, seed=91)
    rng = np.random.default_rng(np.random.PCG64(779))
    _, sc.features, sc.mlp_weights = scenes.draw_neural_appearance(rng, n, 32, 2, 8)
    sc.mlp_hidden, sc.mlp_layers = 32, 2
    cam = scenes.identity_camera(400, 272, 260.0)
    G = np.zeros_like(scenes.upstream_gradient(cam, 5))
    G[:, 3::37, 5::41] = scenes.upstream_gradient(cam, 5)[:, 3::37, 5::41]
    gpu = run_gpu(sc, cam, G)
    _, ref = oracle.render(sc, cam, G)
    for nm in grad_names(sc.app):
        bad = grad_mismatch(getattr(gpu.grads, nm), getattr(ref, nm))
        assert bad.mean() <= 0.002, (nm, int(bad.sum()))
