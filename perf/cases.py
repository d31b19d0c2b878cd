"""Performance cases: the work that users of the library have it do, through its public entry points.

A case is a dict of plain values; `prepare` makes what a program holds before the call (scene, camera, buffers), `run`
makes one pass.  Kinds of passes:

  step     one view of a training step: Renderer.forward, then Renderer.backward with an upstream image gradient
  render   one view without a backward: evaluation, viewer
  train    one training iteration: several views on streams of their own (device-counted, no host wait), each forward and
           backward into gradient buffers of its own, then one fused Adam update of every parameter that sums them
  decode   the separate appearance pass, forward and backward, for given directions
  adam     the fused Adam update of a whole parameter set
  prepass  the viewer's colour prepass of the neural model, once per frame

Scenes follow the distributions of the package's seeded configurations (scenes.py), drawn on the device: a box in front of
an identity camera for small scenes, anisotropic clusters with a background shell for large ones, spread over a depth
range of 1 to 50 for the largest.  Camera angle, upstream gradients and all parameters come from the seed.
"""
import math

import torch

from paper_2609_05255_b200 import api, scenes

SH, NEURAL, SV = api.GS_APP_SH, api.GS_APP_NEURAL, api.GS_APP_SV
APPS = {"sh": SH, "neural": NEURAL, "half": NEURAL, "sv": SV}   # "half": the neural decoder on plain fp16 operands
ROW = {"sh": 45, "neural": 8, "half": 8, "sv": 49}              # view-dependent parameters per Gaussian
ROW_BYTES = {"sh": 180, "neural": 16, "half": 16, "sv": 196}
Y0 = 0.28209479177387814


def listed():
    return [
        # a debugging-size SH scene (the package's configuration 1): launches and host time
        dict(name="step_sh_1k_64", kind="step", app="sh", scene="box", n=1000, width=64, height=64),
        # a small object early in training, half-precision decoder, image and count off every tile size
        dict(name="step_half_20k_333x217", kind="step", app="half", scene="box", n=20011, width=333, height=217),
        # configuration 2: 100k Gaussians, 512 x 512
        dict(name="step_neural_100k_512", kind="step", app="neural", scene="box", n=100_000, width=512, height=512),
        # a NeRF-Synthetic-like scene with Spherical Voronoi appearance, odd sizes
        dict(name="step_sv_300k_799x801", kind="step", app="sv", scene="clusters", n=300_007, width=799, height=801),
        # configuration 3, one view, the explicit baseline model
        dict(name="step_sh_1M_1256x828", kind="step", app="sh", scene="clusters", n=1_000_000, width=1256, height=828),
        # configuration 4, one view: the largest step
        dict(name="step_neural_3M_1080p", kind="step", app="neural", scene="deep", n=3_000_000, width=1920, height=1080),
        # a 1.5M scene rendered at 720p, the setting of the renderer comparison
        dict(name="render_neural_1500k_720p", kind="render", app="neural", scene="clusters", n=1_500_000, width=1280, height=720),
        # configuration 3 as a training iteration: 8 views on 4 streams, one Adam update
        dict(name="train_neural_1M_8views", kind="train", app="neural", scene="clusters", n=1_000_000, width=1256, height=828,
             views=8, streams=4),
        # configuration 5: the separate decode pass
        dict(name="decode_neural_1M", kind="decode", app="neural", n=1_000_000, hidden=16, layers=2, nfeat=8),
        dict(name="decode_sh_3M", kind="decode", app="sh", n=3_000_000, hidden=16, layers=2, nfeat=8),
        # the optimiser on the neural parameter set
        dict(name="adam_neural_1M", kind="adam", app="neural", n=1_000_000),
        # a viewer frame of a 3M scene
        dict(name="prepass_neural_3M", kind="prepass", app="neural", n=3_000_000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _view(rng, most):
    """A scene and an image for it: (scene kind, n, width, height); images grow with the scene."""
    n = _log_int(rng, 1000, most)
    if n <= 150_000:
        kind, side = "box", (64, 512)
    elif n <= 1_500_000:
        kind, side = "clusters", (400, 1000)
    else:
        kind, side = "deep", (700, 1400)
    s = _log_int(rng, *side)
    aspect = rng.uniform(0.75, 1.35)                     # sqrt of width / height: 9:16 to 16:9
    return kind, n, max(33, int(s * aspect)), max(33, int(s / aspect))


def draw(rng):
    kind = rng.choices(["step", "render", "train", "decode", "adam", "prepass"], [50, 15, 10, 15, 5, 5])[0]
    app = rng.choices(["neural", "half", "sh", "sv"], [45, 15, 25, 15])[0]
    if kind in ("step", "render"):
        scene, n, w, h = _view(rng, 3_000_000)
        return dict(kind=kind, app=app, scene=scene, n=n, width=w, height=h)
    if kind == "train":
        scene, n, w, h = _view(rng, 1_000_000)
        views = rng.randint(2, 8)
        return dict(kind=kind, app="neural" if app == "half" else app, scene=scene, n=n, width=w, height=h, views=views,
                    streams=min(views, rng.choice([2, 4])))
    n = _log_int(rng, 10_000, 10_000_000 if kind != "adam" else 3_000_000)
    if kind == "decode":
        hidden, layers, nfeat = 16, 2, 8
        if app == "neural" and rng.random() < 0.3:       # a decoder of another size
            hidden, layers, nfeat = rng.choice([(16, 1, 8), (16, 3, 8), (32, 2, 8), (16, 2, 16)])
            n = min(n, 3_000_000)
        return dict(kind=kind, app=app, n=n, hidden=hidden, layers=layers, nfeat=nfeat)
    if kind == "adam":
        return dict(kind=kind, app="neural" if app == "half" else app, n=n)
    return dict(kind=kind, app="neural", n=n)


# ---- inputs --------------------------------------------------------------------------------------------------------
class _Draw:
    """Random tensors on the device from one seed."""

    def __init__(self, seed):
        self.dev = torch.device("cuda", 0)
        self.gen = torch.Generator(device=self.dev)
        self.gen.manual_seed(seed)

    def normal(self, *shape):
        return torch.randn(shape, device=self.dev, generator=self.gen)

    def uniform(self, lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(shape, device=self.dev, generator=self.gen)

    def index(self, high, *shape):
        return torch.randint(0, high, shape, device=self.dev, generator=self.gen)


def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _geometry(case, d):
    n = case["n"]
    if case["scene"] == "box":
        means = torch.cat([d.uniform(-3.0, 3.0, n, 2), d.uniform(2.0, 8.0, n, 1)], 1)
        if n <= 5000:
            means = torch.cat([d.uniform(-1.0, 1.0, n, 2), d.uniform(2.0, 4.0, n, 1)], 1)
        log_scales, logits = -3.0 + 0.5 * d.normal(n, 3), d.normal(n)
    else:
        deep = case["scene"] == "deep"
        clusters = 256 if deep else 64
        shell = n // 10
        if deep:
            radius = torch.exp(d.uniform(math.log(0.5), math.log(45.0), clusters, 1))
        else:
            radius = 2.0 * d.uniform(0.0, 1.0, clusters, 1) ** (1.0 / 3.0)
        centres = _unit(d.normal(clusters, 3)) * radius
        w, x, y, z = _unit(d.normal(clusters, 4)).unbind(1)
        rot = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                           2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                           2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).reshape(clusters, 3, 3)
        spread = rot * (0.3 * torch.exp(0.5 * d.normal(clusters, 1, 3)))
        member = d.index(clusters, n)                    # a draw per Gaussian: no spatial order in memory
        means = centres[member] + (spread[member] @ d.normal(n, 3, 1)).squeeze(2)
        far = torch.rand((n,), device=d.dev, generator=d.gen) < shell / n
        means = torch.where(far[:, None], 20.0 * _unit(d.normal(n, 3)), means)
        log_scales = (-4.5 + 0.8 * d.normal(n, 3)) if deep else (-4.0 + 0.7 * d.normal(n, 3))
        logits = 1.5 * d.normal(n)
    return means.contiguous(), log_scales.contiguous(), d.normal(n, 4), logits.contiguous()


def _appearance(case, d):
    """The appearance members of a DeviceScene, as keyword arguments."""
    n, app = case["n"], case["app"]
    base = Y0 * (0.5 + 0.1 * d.normal(n, 3))
    if app == "sh":
        return dict(base_color=base, sh_rest=0.05 * d.normal(n, 15, 3))
    if app == "sv":
        lattice = torch.from_numpy(scenes.fibonacci_sites(7)).to(d.dev, torch.float32)
        sites = torch.cat([0.15 * d.normal(n, 7, 3), (lattice + 0.25 * d.normal(n, 7, 3)) * d.uniform(0.5, 2.0, n, 7, 1),
                           0.5 + 0.5 * d.normal(n, 7, 1)], 2)
        return dict(base_color=base, sv_sites=sites.contiguous())
    hidden, layers, nfeat = case.get("hidden", 16), case.get("layers", 2), case.get("nfeat", 8)
    shapes = [(hidden, 32)] + [(hidden, hidden)] * (layers - 1) + [(3, hidden)]
    weights = torch.cat([d.uniform(-1.0, 1.0, o * i) * math.sqrt(6.0 / (i + o)) for o, i in shapes])
    return dict(base_color=base, features=(0.1 * d.normal(n, nfeat)).half(), mlp_weights=weights.half(), mlp_hidden=hidden,
                mlp_layers=layers, num_features=nfeat, decoder_precision=api.GS_DECODER_HALF if app == "half" else api.GS_DECODER_SPLIT)


def _cameras(case, d, count):
    w, h = case["width"], case["height"]
    if case["scene"] == "box":
        focal = max(w, h)
        return [api.make_camera(scenes.identity_camera(w, h, focal * (1.0 + 0.05 * k), background=(0.1, 0.2, 0.3))) for k in range(count)]
    turn = float(d.uniform(0.0, 2.0 * math.pi, 1))
    return [api.make_camera(scenes.orbit_camera(w, h, turn + 2.0 * math.pi * k / count)) for k in range(count)]


# (column count, learning rate) of every parameter; rates at the end of their schedules
RATES = {"means": (3, 1.6e-6), "log_scales": (3, 5e-5), "quats": (4, 1e-5), "opacity_logits": (1, 5e-4), "base_color": (3, 2.5e-5),
         "sh_rest": (45, 1.25e-6), "features": (8, 8e-5), "mlp_weights": (1, 3e-5), "sv_sites": (49, 2e-5)}
GEOMETRY = ["means", "log_scales", "quats", "opacity_logits", "base_color"]
VIEW_PART = {"sh": ["sh_rest"], "neural": ["features", "mlp_weights"], "half": ["features", "mlp_weights"], "sv": ["sv_sites"]}


def _names(case):
    return GEOMETRY + VIEW_PART[case["app"]]


def _outputs(grads, case):
    return {name: getattr(grads, name) for name in _names(case)}


def prepare(case, seed):
    d = _Draw(seed)
    ctx = api.Context(0)
    s = dict(case=case, ctx=ctx)
    if case["kind"] == "adam":
        _prepare_adam(s, d, {name: ((case["n"] if name != "mlp_weights" else 816), RATES[name][0]) for name in _names(case)})
        return s
    if case["kind"] in ("decode", "prepass"):
        n, z = case["n"], torch.zeros((1, 4), device=d.dev)
        means = d.normal(n, 3) if case["kind"] == "prepass" else z
        logits = 1.5 * d.normal(n) if case["kind"] == "prepass" else z[0]
        s["scene"] = scene = api.DeviceScene(means, z, z, logits, app=APPS[case["app"]], active_degree=3, **_appearance(case, d))
        if case["kind"] == "prepass":
            s["preact"] = torch.empty((n, 16), device=d.dev, dtype=torch.float16)
            api.gs_neural_fold(ctx, scene, s["preact"])
            s["cam"] = api.make_camera(scenes.orbit_camera(1256, 828, float(d.uniform(0.0, 6.28, 1))))
            s["rgba"] = torch.empty((n, 4), device=d.dev, dtype=torch.uint8)
        else:
            s["dirs"], s["upstream"] = _unit(d.normal(n, 3)).contiguous(), d.normal(n, 3)
            s["color"], s["g_dirs"] = torch.empty((n, 3), device=d.dev), torch.empty((n, 3), device=d.dev)
            s["grads"] = api.alloc_grads_for(scene, d.dev)
        return s
    s["scene"] = scene = api.DeviceScene(*_geometry(case, d), app=APPS[case["app"]], active_degree=3, **_appearance(case, d))
    views = case.get("views", 1)
    s["cams"] = _cameras(case, d, views)
    w, h = case["width"], case["height"]
    # instance capacity: what the views need, with the slack of a scene that moves
    probe = api.alloc_projected(scene.n, d.dev)
    capacity = int(1.1 * max(api.gs_preprocess(ctx, scene, c, probe) for c in s["cams"])) + 4096
    del probe
    s["upstream"] = d.normal(views, 3, h, w)
    if case["kind"] != "train":
        s["renderer"] = api.Renderer(ctx, scene.n, w, h, scene.app, capacity)
        return s
    lanes = case["streams"]
    s["lanes"] = [torch.cuda.Stream(d.dev) for _ in range(lanes)]
    s["ctxs"] = [ctx] + [api.Context(0) for _ in range(lanes - 1)]
    s["renderers"] = [api.Renderer(c, scene.n, w, h, scene.app, capacity) for c in s["ctxs"]]
    s["images"] = [torch.empty((3, h, w), device=d.dev) for _ in range(views)]
    s["grads"] = [api.alloc_grads(scene.n, scene.app, d.dev) for _ in range(views)]
    _prepare_adam(s, d, {name: (getattr(scene, name).numel() // RATES[name][0], RATES[name][0]) for name in _names(case)})
    return s


def _prepare_adam(s, d, shapes):
    """Masters, moments (of an optimiser that has run for a while) and the argument list of the update."""
    case, scene, grads = s["case"], s.get("scene"), s.get("grads")
    s["step"], s["adam"], s["updated"] = 1000, [], {}
    for name, (rows, cols) in shapes.items():
        stored = getattr(scene, name) if scene else d.normal(rows, cols)
        master = stored.float().contiguous() if stored.dtype != torch.float32 else stored
        grad = getattr(grads[0], name) if grads else 1e-3 * d.normal(rows, cols)
        scale = 1.0 if grads else 1e-3
        m, v = 0.1 * scale * d.normal(rows, cols), (scale * d.uniform(0.5, 1.5, rows, cols)) ** 2
        half = None
        if name in ("features", "mlp_weights"):
            half = stored if scene else torch.empty((rows, cols), device=d.dev, dtype=torch.float16)
        s["adam"].append(api.AdamTensor(master, grad, m, v, [RATES[name][1]] * cols, 0.9, 0.99 if name == "mlp_weights" else 0.999,
                                        1e-15, half_copy=half, more_grads=[getattr(g, name) for g in grads[1:]] if grads else ()))
        s["updated"].update({name: master, name + "_m": m, name + "_v": v})
        if half is not None:
            s["updated"][name + "_half"] = half


# ---- one pass ------------------------------------------------------------------------------------------------------
def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "step":
        r, cam = s["renderer"], s["cams"][0]
        image = r.forward(s["scene"], cam)
        grads = r.backward(s["scene"], cam, s["upstream"][0])
        return dict(image=image, final_T=r.final_T, n_contrib=r.n_contrib, **_outputs(grads, case))
    if kind == "render":
        r = s["renderer"]
        image = r.forward(s["scene"], s["cams"][0])
        return dict(image=image, final_T=r.final_T, n_contrib=r.n_contrib)
    if kind == "train":
        main = torch.cuda.current_stream()
        lanes, renderers = s["lanes"], s["renderers"]
        for lane in lanes:
            lane.wait_stream(main)
        for v, cam in enumerate(s["cams"]):
            r, lane = renderers[v % len(lanes)], lanes[v % len(lanes)]
            r.image, r.grads = s["images"][v], s["grads"][v]
            r.forward_async(s["scene"], cam, stream=lane)
            r.backward(s["scene"], cam, s["upstream"][v], stream=lane)
        for lane in lanes:
            main.wait_stream(lane)
        s["step"] += 1
        api.gs_adam_step(ctx, s["adam"], s["step"])
        return dict(images=s["images"], **s["updated"])
    if kind == "decode":
        api.gs_appearance_forward(ctx, s["scene"], s["dirs"], s["color"])
        api.gs_appearance_backward(ctx, s["scene"], s["dirs"], s["upstream"], s["grads"], s["g_dirs"])
        names = ["base_color"] + VIEW_PART[case["app"]]
        return dict(color=s["color"], g_dirs=s["g_dirs"], **{name: getattr(s["grads"], name) for name in names})
    if kind == "adam":
        s["step"] += 1
        api.gs_adam_step(ctx, s["adam"], s["step"])
        return s["updated"]
    api.gs_neural_prepass(ctx, s["scene"], s["preact"], s["cam"], s["rgba"])
    return s["rgba"]


# ---- what a pass cannot do without -----------------------------------------------------------------------------------
def _adam_bytes(case, grad_sets):
    total = 0
    for name in _names(case):
        count = (case["n"] if name != "mlp_weights" else 816) * (RATES[name][0] if name != "mlp_weights" else 1)
        total += count * (24 + 4 * grad_sets + (2 if name in ("features", "mlp_weights") else 0))
    return total


def work(case):
    kind, n, app = case["kind"], case["n"], case["app"]
    macs = 816 if app in ("neural", "half") else 45 if app == "sh" else 140
    if kind == "adam":
        return dict(bytes=_adam_bytes(case, 1), flops=12 * n * sum(RATES[k][0] for k in _names(case)))
    if kind == "prepass":
        return dict(bytes=64 * n, flops=2 * 560 * n)
    if kind == "decode":
        if app in ("neural", "half"):
            h, l, nf = case["hidden"], case["layers"], case["nfeat"]
            macs = 32 * h + (l - 1) * h * h + 3 * h
            row, row_grad = 2 * nf, 4 * nf
        else:
            row = row_grad = ROW_BYTES[app]
        # forward: direction, base colour, row in, colour out; backward: the same and dL/dcolour in, three gradients out
        return dict(bytes=n * (36 + row + 36 + row + 24 + row_grad), flops=n * 8 * macs)
    # a view: parameters in; image, transmittance and position out; about 64 composited pairs per pixel, of 18 operations
    # forward and 45 backward; per Gaussian 400 operations of projection
    pixels = case["width"] * case["height"]
    views = case.get("views", 1)
    bytes_, flops = n * (56 + ROW_BYTES[app]) + 20 * pixels, n * (400 + 2 * macs) + 64 * 18 * pixels
    if kind != "render":
        bytes_ += n * (56 + 4 * ROW[app]) + 20 * pixels       # gradients out; upstream, transmittance and position in
        flops += 64 * 45 * pixels + n * 400
    total = dict(bytes=views * bytes_, flops=views * flops)
    if kind == "train":
        total["bytes"] += _adam_bytes(case, views)
    return total


def tolerance(case):
    kind, app = case["kind"], case["app"]
    if kind == "adam":
        return dict(rel=1e-5, max=1e-3)          # one chain of 32-bit multiply-adds per element
    if kind == "prepass":
        return dict(differ=0.01)                 # half-precision operands: a texel may round the other way
    if kind == "decode":
        if app in ("sh", "sv"):
            return dict(rel=1e-5, max=1e-2)
        # split operands carry 22 bits; in a few of a million Gaussians a hidden unit at its kink takes the other branch
        return dict(rel=3e-4 if app == "neural" else 5e-3, max=0.9)
    # 32-bit sums over hundreds of pairs per pixel and thousands of pixels per Gaussian, of both signs; a pair at the
    # threshold alpha = 1/255 may fall on either side
    return dict(rel=5e-3 if app == "half" else 5e-4, max=0.5, differ=1e-3)
