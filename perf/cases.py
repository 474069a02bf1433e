"""The work that a user of the rasterizer has it do, as cases to be timed and compared.

Every case goes through the public entry points (render, rasterize, Frame, FrameBatch, SceneBatch,
Trainer, Loss, DensityControl).  Scenes follow the distributions of ``synthetic`` and are drawn on the
GPU from the seed: "box" (config 1), "cluster" (configs 2 and 5) and "unbounded" (configs 3 and 4).
"""
from __future__ import annotations

import math
import random
from types import SimpleNamespace

import numpy as np
import torch

from paper_2308_04079_gb300 import Frame, FrameBatch, GaussianTensors, make_config, rasterize, render
from paper_2308_04079_gb300.batching import Scene, SceneBatch
from paper_2308_04079_gb300.density import DensityControl, DensitySchedule
from paper_2308_04079_gb300.training import GaussianModel, Loss, Trainer

BLACK = (0.0, 0.0, 0.0)
RESOLUTIONS = ((640, 480), (1280, 720), (1600, 900), (1920, 1080))
PARAMS = ("means", "log_scales", "quats", "logit_opacities", "sh")


def listed():
    return [
        # a thumbnail of a few Gaussians: launches and host calls are all there is
        dict(name="render_1k_128", kind="render", scene="box", n=1000, degree=0, width=128, height=128, tile="16x16"),
        # an interactive preview: a ragged image, low SH degree, small tiles
        dict(name="render_60k_813x611", kind="render", scene="cluster", n=60_007, degree=1, width=813, height=611,
             tile="8x8"),
        # the real-time viewer on a large captured scene
        dict(name="render_3m_1080p", kind="render", scene="unbounded", n=3_000_000, degree=3, width=1920, height=1080,
             tile="16x16"),
        # a crop of a view, differentiated through autograd
        dict(name="rasterize_5k_64", kind="rasterize", scene="cluster", n=5000, degree=3, width=64, height=64,
             tile="16x16"),
        # one view of a small scene through autograd, in someone's own training loop
        dict(name="rasterize_200k_1080p", kind="rasterize", scene="cluster", n=200_000, degree=3, width=1920,
             height=1080, tile="16x16"),
        # the headline frame: forward and backward of a large scene through the stage calls
        dict(name="frame_3m_1080p", kind="frame", scene="unbounded", n=3_000_000, degree=3, width=1920, height=1080,
             tile="16x16", isotropic=False, grad_limit=0),
        # the ablation variants (isotropic, Limited-BW) at a ragged size and the middle tile shape
        dict(name="frame_variant_500k_1601x901", kind="frame", scene="unbounded", n=500_003, degree=2, width=1601,
             height=901, tile="16x8", isotropic=True, grad_limit=10),
        # one training iteration, density statistics among it, at a size of the early optimisation
        dict(name="train_150k_979x546", kind="train", scene="cluster", n=150_000, degree=3, width=979, height=546),
        # sixteen views of one scene as one batch, gradients summed
        dict(name="batch_1m_16views", kind="batch", scene="unbounded", n=1_000_000, degree=3, views=16, shrink=1.0),
        # several scenes of uneven size, the whole step replayed as one CUDA graph
        dict(name="scenes_4x3", kind="scenes", scene="cluster", n=50_000, n_max=800_000, degree=3, scenes=4, views=3,
             shrink=1.0),
        # the training loss and its image gradient
        dict(name="loss_1080p", kind="loss", width=1920, height=1080),
        # a refinement: prune, clone and split parameters and moments
        dict(name="refine_1m", kind="refine", n=1_000_000, degree=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(("render", "render", "rasterize", "frame", "frame", "train", "batch", "scenes", "loss", "refine"))
    if kind == "loss":
        return dict(kind=kind, width=_log_int(rng, 64, 1920), height=_log_int(rng, 64, 1080))
    if kind == "refine":
        return dict(kind=kind, n=_log_int(rng, 2000, 1_000_000), degree=rng.choice((0, 1, 2, 3)))
    scene = rng.choice(("cluster", "unbounded"))
    if kind == "batch":
        return dict(kind=kind, scene=scene, n=_log_int(rng, 20_000, 600_000), degree=rng.choice((1, 3)),
                    views=rng.randint(2, 12), shrink=rng.uniform(0.25, 1.0))
    if kind == "scenes":
        lo = _log_int(rng, 5000, 50_000)
        return dict(kind=kind, scene=scene, n=lo, n_max=lo * rng.randint(2, 10), degree=3, scenes=rng.randint(2, 4),
                    views=rng.randint(1, 3), shrink=rng.uniform(0.25, 1.0))
    width = _log_int(rng, 64, 1920)
    size = dict(kind=kind, scene=scene, width=width, height=min(1080, max(48, int(width * rng.uniform(0.5, 1.0)))))
    if kind == "train":
        return dict(size, n=_log_int(rng, 2000, 300_000), degree=3)
    size.update(n=_log_int(rng, 1000, 2_000_000 if kind == "frame" else 600_000), degree=rng.choice((0, 1, 2, 3, 3, 3)),
                tile=rng.choice(("16x16", "16x16", "16x8", "8x8")))
    if kind == "frame":
        size.update(isotropic=rng.random() < 0.25, grad_limit=rng.choice((0, 0, 0, 10)))
    return size


# ---- inputs ---------------------------------------------------------------------------------


def _look_at(eye, width, height, fov_x_deg=60.0):
    eye = np.asarray(eye, np.float64)
    fwd = -eye / np.linalg.norm(eye)
    right = np.cross([0.0, 1.0, 0.0], fwd)
    right /= np.linalg.norm(right)
    R = np.stack([right, np.cross(fwd, right), fwd]).astype(np.float32).astype(np.float64)
    t = (-R @ eye).astype(np.float32).astype(np.float64)
    f = float(np.float32(0.5 * width / math.tan(math.radians(fov_x_deg) / 2)))
    return SimpleNamespace(width=width, height=height, fx=f, fy=f, cx=width / 2.0, cy=height / 2.0, R=R, t=t,
                           near=float(np.float32(0.2)))


def _orbit(rng, scene, width, height):
    radius = {"box": 4.0, "cluster": 8.0, "unbounded": 3.0}[scene]
    az, el = rng.uniform(0.0, 2.0 * math.pi), math.radians(rng.uniform(-30.0, 30.0))
    eye = (radius * math.cos(el) * math.sin(az), -radius * math.sin(el), -radius * math.cos(el) * math.cos(az))
    return _look_at(eye, width, height)


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _ball(gen, n, r_in, r_out):
    d = torch.nn.functional.normalize(torch.randn(n, 3, generator=gen, device="cuda"), dim=1)
    u = torch.rand(n, 1, generator=gen, device="cuda")
    return d * (r_in ** 3 + u * (r_out ** 3 - r_in ** 3)) ** (1.0 / 3.0)


def _rotations(q):
    """Rotation matrices [N, 3, 3] of unit quaternions (r, i, j, k)."""
    r, i, j, k = q.unbind(1)
    return torch.stack([1 - 2 * (j * j + k * k), 2 * (i * j - r * k), 2 * (i * k + r * j),
                        2 * (i * j + r * k), 1 - 2 * (i * i + k * k), 2 * (j * k - r * i),
                        2 * (i * k - r * j), 2 * (j * k + r * i), 1 - 2 * (i * i + j * j)], 1).view(-1, 3, 3)


def _scene(case, seed, n=None, isotropic=False):
    """Activated parameters as a dict of float32 CUDA tensors."""
    n = case["n"] if n is None else n
    gen = _generator(seed)
    rand = lambda *s: torch.rand(*s, generator=gen, device="cuda")      # noqa: E731
    randn = lambda *s: torch.randn(*s, generator=gen, device="cuda")    # noqa: E731
    logit = randn(n)
    if case["scene"] == "box":
        means, log_s = rand(n, 3) * 2 - 1, 0.5 * randn(n, 3) - 3.0
    elif case["scene"] == "cluster":
        centres, stds = 6.0 * rand(64, 3) - 3.0, 0.05 + 0.45 * rand(64, 3)
        frames = _rotations(torch.nn.functional.normalize(randn(64, 4), dim=1))
        which = torch.randint(0, 64, (n,), generator=gen, device="cuda")
        means = centres[which] + torch.einsum("nij,nj->ni", frames[which], stds[which] * randn(n, 3))
        log_s = randn(n, 3) - 4.0
    else:
        inner = int(round(0.8 * n))
        means = torch.cat([_ball(gen, inner, 0.0, 1.0), _ball(gen, n - inner, 5.0, 50.0)])
        log_s = randn(n, 3)
        log_s[:inner] -= 5.0
        log_s[inner:] -= 2.0
        logit *= 1.5
    sh = 0.05 * randn(n, (case["degree"] + 1) ** 2, 3)
    sh[:, 0] = rand(n, 3) * (2.0 * math.sqrt(math.pi) if case["degree"] == 0 else 1.0)
    quats = torch.nn.functional.normalize(randn(n, 4), dim=1)
    p = dict(means=means, scales=torch.exp(log_s), quats=quats, opacities=torch.sigmoid(logit), sh=sh)
    if isotropic:
        p.update(scales=p["scales"][:, 0].contiguous(), quats=None)
    return p


def _tensors(p, degree):
    return GaussianTensors(p["means"], p["scales"], p["quats"], p["opacities"], p["sh"], degree)


def _image_grad(seed, height, width):
    return torch.randn(3, height, width, generator=_generator(seed), device="cuda")


def _photo(seed, height, width):
    """A smooth image in [0, 1] with some texture."""
    gen = _generator(seed)
    low = torch.rand(1, 3, 9, 16, generator=gen, device="cuda")
    img = torch.nn.functional.interpolate(low, size=(height, width), mode="bicubic", align_corners=False)[0]
    return (img + 0.05 * torch.randn(3, height, width, generator=gen, device="cuda")).clamp(0, 1).contiguous()


def _cfg(case):
    w, h = (int(x) for x in case["tile"].split("x"))
    return make_config(tile=(w, h), isotropic=bool(case.get("isotropic")), grad_limit=case.get("grad_limit", 0))


def _view_sizes(count, shrink):
    for i in range(count):      # uneven, in no order of size
        w, h = RESOLUTIONS[(3 * i + i // 4) % len(RESOLUTIONS)]
        yield max(48, int(w * shrink)), max(48, int(h * shrink))


def _model(case, seed):
    """A model in the middle of its training: raw parameters and moments of the size of its gradients."""
    p = _scene(case, seed)
    m = GaussianModel(p["means"], torch.log(p["scales"]), p["quats"], torch.logit(p["opacities"], eps=1e-6), p["sh"],
                      case["degree"])
    m.scales, m.opacities = torch.exp(m.log_scales), torch.sigmoid(m.logit_opacities)
    gen = _generator(seed + 1)
    for k in PARAMS:
        t = getattr(m, k)
        size = 1e-5 * (0.5 + torch.rand(t.shape, generator=gen, device="cuda"))
        m.moments[k] = (0.3 * size * torch.randn(t.shape, generator=gen, device="cuda"), size * size)
    return m


def _density_inputs(case, seed):
    """Parameters, moments and gradient statistics at a refinement (as synthetic.density_state).  What
    the decisions are made from is the same set of rows for every seed, in another order, so that as many
    rows come out."""
    n, gen = case["n"], _generator(17)
    rand = lambda *s: torch.rand(*s, generator=gen, device="cuda")      # noqa: E731
    randn = lambda *s: torch.randn(*s, generator=gen, device="cuda")    # noqa: E731
    log_scales, logit = randn(n, 3) - 4.0, 2.5 * randn(n) - 1
    count = torch.randint(0, 40, (n,), generator=gen, device="cuda").float()
    accum = count * torch.exp(0.8 * randn(n) + math.log(2e-4))
    radius = torch.floor(-8.0 * torch.log1p(-rand(n))) * (count > 0)
    gen.manual_seed(seed)
    rows = torch.randperm(n, generator=gen, device="cuda")
    p = dict(means=2 * rand(n, 3) - 1, log_scales=log_scales[rows], quats=randn(n, 4), logit_opacities=logit[rows],
             sh=0.3 * randn(n, (case["degree"] + 1) ** 2, 3))
    m = {k: 1e-3 * randn(*t.shape) for k, t in p.items()}
    v = {k: 1e-6 * rand(*t.shape) for k, t in p.items()}
    return p, m, v, accum[rows], count[rows], radius[rows]


def prepare(case, seed):
    kind, rng = case["kind"], random.Random(seed)
    s = SimpleNamespace(kind=kind, case=case, seed=seed)
    if kind == "loss":
        w, h = case["width"], case["height"]
        s.loss, s.img, s.target = Loss(w, h), _photo(2 * seed, h, w), _photo(2 * seed + 1, h, w)
        s.grad = torch.empty_like(s.img)
        return s
    if kind == "refine":
        s.inputs = _density_inputs(case, seed)
        s.gen = _generator(seed)
        return s
    if kind == "train":
        s.camera = _orbit(rng, case["scene"], case["width"], case["height"])
        s.target = _photo(seed + 2, case["height"], case["width"])
        s.model = _model(case, seed)
        # between two refinements: statistics gathered, none due
        between = DensitySchedule(start=1 << 30, reset_every=0)
        s.trainer = Trainer(s.model, density=DensityControl(s.model, extent=8.8, schedule=between))
        s.trainer.iteration = 1000
        return s
    if kind == "batch":
        s.g = _tensors(_scene(case, seed), case["degree"]).prepared()
        cams = [_orbit(rng, case["scene"], w, h) for w, h in _view_sizes(case["views"], case["shrink"])]
        s.dimgs = [_image_grad(seed + 100 + i, c.height, c.width) for i, c in enumerate(cams)]
        cfg = make_config()
        probe = FrameBatch([Frame(s.g.n, c, cfg) for c in cams], [s.g] * len(cams))
        probe.ensure_binned()
        # the workspaces a program keeps: sized to the views' instance counts
        s.frames = [Frame(s.g.n, c, cfg, capacity=int(f.last_status.num_instances * 1.15) + 4096)
                    for c, f in zip(cams, probe.frames)]
        s.batch = FrameBatch(s.frames, [s.g] * len(cams))
        s.outs = s.batch.outputs()
        s.grads = s.frames[0].new_grads(s.g)
        return s
    if kind == "scenes":
        scenes, k = [], max(1, case["scenes"] - 1)
        for i in range(case["scenes"]):
            n = int(case["n"] * (case["n_max"] / case["n"]) ** (i / k))
            g = _tensors(_scene(case, seed + i, n), case["degree"]).prepared()
            cams = [_orbit(rng, case["scene"], w, h) for w, h in _view_sizes(case["views"], case["shrink"])]
            scenes.append(Scene(g, cams, [_image_grad(seed + 100 + 10 * i + j, c.height, c.width)
                                          for j, c in enumerate(cams)]))
        s.scenes, s.batch = scenes, SceneBatch(scenes)
        s.batch.capture()
        return s
    cam = s.camera = _orbit(rng, case["scene"], case["width"], case["height"])
    s.cfg = _cfg(case)
    p = s.params = _scene(case, seed, isotropic=bool(case.get("isotropic")))
    if kind == "render":
        s.g = _tensors(p, case["degree"])
        s.frame = render(s.g, cam, BLACK, s.cfg)[3]     # the viewer's workspace, grown by an earlier view
        return s
    s.dimg = _image_grad(seed + 3, cam.height, cam.width)
    if kind == "rasterize":
        s.leaves = [p[k].requires_grad_() for k in ("means", "scales", "quats", "opacities", "sh")]
        s.settings = dict(frame=render(_tensors(p, case["degree"]), cam, BLACK, s.cfg)[3])
        return s
    s.g = _tensors(p, case["degree"]).prepared()
    probe = Frame(s.g.n, cam, s.cfg)
    probe.ensure_binned(s.g)
    s.frame = Frame(s.g.n, cam, s.cfg, capacity=int(probe.last_status.num_instances * 1.15) + 4096)
    s.outs = s.frame.outputs()
    s.grads = s.frame.new_grads(s.g)
    return s


def _kept(d):
    return {k: t for k, t in d.items() if t is not None}


def run(s):
    if s.kind == "render":
        img, T, last, s.frame = render(s.g, s.camera, BLACK, s.cfg, frame=s.frame)
        return dict(image=img, T=T, last=last)
    if s.kind == "rasterize":
        img = rasterize(*s.leaves, s.case["degree"], s.camera, BLACK, s.cfg, s.settings)
        grads = torch.autograd.grad(img, s.leaves, s.dimg)
        return dict(image=img, grads=list(grads), mean2d=s.settings["mean2d_grad"])
    if s.kind == "frame":
        f = s.frame
        f.preprocess(s.g)
        f.bin_sort()
        f.render_forward(BLACK, *s.outs)
        f.render_backward(s.g, BLACK, s.dimg, s.outs[1], s.outs[2], s.grads)
        return dict(image=s.outs[0], T=s.outs[1], last=s.outs[2], grads=_kept(s.grads))
    if s.kind == "batch":
        b = s.batch
        b.preprocess()
        b.bin_sort()
        b.render_forward(BLACK, s.outs)
        b.render_backward(BLACK, s.dimgs, s.outs, [s.grads] * len(s.outs))
        return dict(views=[list(o) for o in s.outs], grads=_kept(s.grads))
    if s.kind == "scenes":
        s.batch.replay()
        return dict(views=[list(o) for o in s.batch.outs], grads=[_kept(s.batch.scene_grads(x)) for x in s.scenes])
    if s.kind == "train":
        loss = s.trainer.step(s.camera, s.target)
        m, d = s.model, s.trainer.density
        return dict(loss=loss, params={k: getattr(m, k) for k in PARAMS}, moments={k: list(m.moments[k]) for k in PARAMS},
                    stats=[d.grad_accum, d.grad_count, d.max_radius])
    if s.kind == "loss":
        return dict(loss=s.loss(s.img, s.target, s.grad), grad=s.grad)
    # refine: the statistics that training gathered, and a model whose tensors the refinement replaces
    p, m, v, accum, count, radius = s.inputs
    model = GaussianModel(p["means"], p["log_scales"], p["quats"], p["logit_opacities"], p["sh"], s.case["degree"],
                          moments={k: (m[k], v[k]) for k in PARAMS})
    dc = DensityControl(model, extent=3.0)
    dc.grad_accum, dc.grad_count, dc.max_radius = accum, count, radius
    rows = dc.refine(size_pruning=True, generator=s.gen.manual_seed(s.seed))
    return dict(rows=rows, params={k: getattr(model, k) for k in PARAMS},
                moments={k: list(model.moments[k]) for k in PARAMS}, scales=model.scales, opacities=model.opacities)


def _floats(case, isotropic=False):
    """Floats of one Gaussian's parameters."""
    return 3 * (case["degree"] + 1) ** 2 + (5 if isotropic else 11)


def work(case):
    """Bytes: every input read once, every output written once.  Flops: per Gaussian the projection, colour
    and (backward) their chain rule; per pixel one blend of ten splats, the least a covered pixel takes."""
    kind = case["kind"]
    if kind == "loss":
        px = case["width"] * case["height"] * 3
        return dict(bytes=12 * px, flops=px * (8 * 2 * 22 + 60))
    n, f = case["n"], _floats(case, bool(case.get("isotropic")))
    if kind == "refine":
        return dict(bytes=2 * 4 * n * (3 * f + 6), flops=20 * n)
    fwd, bwd = 400 + 6 * (case["degree"] + 1) ** 2, 800 + 12 * (case["degree"] + 1) ** 2
    mean_px = 0.25 * sum(w * h for w, h in RESOLUTIONS) * case.get("shrink", 1.0) ** 2
    if kind == "batch":
        px = mean_px * case["views"]
        return dict(bytes=4 * (n * (2 * f + 2) + 8 * px), flops=case["views"] * n * (fwd + bwd) + px * 10 * 60)
    if kind == "scenes":
        k = max(1, case["scenes"] - 1)
        total = sum(int(n * (case["n_max"] / n) ** (i / k)) for i in range(case["scenes"]))
        px = mean_px * case["views"] * case["scenes"]
        return dict(bytes=4 * (total * (2 * f + 2) + 8 * px),
                    flops=case["views"] * total * (fwd + bwd) + px * 10 * 60)
    px = case["width"] * case["height"]
    if kind == "render":
        return dict(bytes=4 * (n * f + 5 * px), flops=n * fwd + px * 10 * 20)
    if kind == "train":   # parameters and moments read and written, activations, image gradient
        return dict(bytes=4 * (n * (6 * f + 4 + 6) + 3 * px), flops=n * (fwd + bwd + 15 * f) + px * (10 * 60 + 3 * 410))
    return dict(bytes=4 * (n * (2 * f + 2) + (6 if kind == "rasterize" else 8) * px),
                flops=n * (fwd + bwd) + px * 10 * 60)


# ---- the same in 64 bits, by definition -------------------------------------------------------


def exact(case, seed):
    kind = case["kind"]
    if kind == "loss":
        return _exact_loss(prepare(case, seed))
    if kind == "refine":
        return _exact_refine(prepare(case, seed))
    if kind not in ("render", "rasterize", "frame") or case["n"] * case["width"] * case["height"] > 30_000_000:
        return None     # every pixel against every Gaussian: small frames only
    if case.get("grad_limit"):
        return None
    rng = random.Random(seed)
    cam = _orbit(rng, case["scene"], case["width"], case["height"])
    p = _scene(case, seed, isotropic=bool(case.get("isotropic")))
    dimg = None if kind == "render" else _image_grad(seed + 3, cam.height, cam.width)
    img, T, grads, mean2d = _exact_frame(p, case, cam, dimg)
    if kind == "render":
        return dict(image=img, T=T, last=None)
    if kind == "rasterize":
        return dict(image=img, grads=[grads[k] for k in ("means", "scales", "quats", "opacities", "sh")], mean2d=mean2d)
    return dict(image=img, T=T, last=None, grads=dict(_kept(grads), mean2d=mean2d))


def _sh_basis(d, degree):
    x, y, z = d.unbind(1)
    Y = [torch.full_like(x, 0.5 / math.sqrt(math.pi))]
    if degree > 0:
        c = math.sqrt(3 / (4 * math.pi))
        Y += [-c * y, c * z, -c * x]
    if degree > 1:
        a, b = math.sqrt(15 / math.pi) / 2, math.sqrt(5 / math.pi) / 4
        Y += [a * x * y, -a * y * z, b * (3 * z * z - 1), -a * x * z, a / 2 * (x * x - y * y)]
    if degree > 2:
        a, b = math.sqrt(35 / (2 * math.pi)) / 4, math.sqrt(105 / math.pi)
        c, e = math.sqrt(21 / (2 * math.pi)) / 4, math.sqrt(7 / math.pi) / 4
        Y += [-a * y * (3 * x * x - y * y), b / 2 * x * y * z, -c * y * (5 * z * z - 1), e * z * (5 * z * z - 3),
              -c * x * (5 * z * z - 1), b / 4 * z * (x * x - y * y), -a * x * (x * x - 3 * y * y)]
    return torch.stack(Y, 1)


def _exact_frame(p, case, cam, dimg):
    tile_w, tile_h = (int(v) for v in case["tile"].split("x"))
    iso = p["quats"] is None
    leaves = {k: t.double().requires_grad_() for k, t in p.items() if t is not None}
    mu, sh = leaves["means"], leaves["sh"]
    R, t = (torch.tensor(np.asarray(a), dtype=torch.float64, device="cuda") for a in (cam.R, cam.t))
    cc = mu @ R.T + t
    x, y, z = cc.unbind(1)
    fx, fy, W, H = cam.fx, cam.fy, cam.width, cam.height
    guard = float(np.float32(1.3))
    vis = (z > cam.near) & ((x / z).abs() <= guard * 0.5 * W / fx) & ((y / z).abs() <= guard * 0.5 * H / fy)
    zs = torch.where(vis, z, torch.ones_like(z))
    uv = torch.stack([fx * x / zs + cam.cx, fy * y / zs + cam.cy], 1)
    zero = torch.zeros_like(zs)
    J = torch.stack([torch.stack([fx / zs, zero, -fx * x / zs ** 2], 1),
                     torch.stack([zero, fy / zs, -fy * y / zs ** 2], 1)], 1)
    if iso:
        M = leaves["scales"][:, None, None] * torch.eye(3, dtype=torch.float64, device="cuda")
    else:
        M = _rotations(torch.nn.functional.normalize(leaves["quats"], dim=1)) * leaves["scales"][:, None, :]
    V = J @ R @ M
    S = V @ V.transpose(1, 2) + float(np.float32(0.3)) * torch.eye(2, dtype=torch.float64, device="cuda")
    A, B, C = S[:, 0, 0], S[:, 0, 1], S[:, 1, 1]
    det = A * C - B * B
    lam = 0.5 * (A + C) + torch.sqrt((0.5 * (A - C)) ** 2 + B * B)
    rad = torch.ceil(3.0 * torch.sqrt(lam)).detach()
    campos = -R.T @ t
    colour = (torch.einsum("nk,nkc->nc", _sh_basis(torch.nn.functional.normalize(mu - campos, dim=1), case["degree"]), sh)
              .clamp(min=0))
    # front to back: by the 32-bit depth, ties by index
    order = torch.sort(z.detach().float(), stable=True)[1]
    order = order[vis[order]]
    splat_uv = uv[order]
    splat_uv.retain_grad()
    u, v = splat_uv[:, 0], splat_uv[:, 1]
    px = torch.arange(W, device="cuda", dtype=torch.float64)
    py = torch.arange(H, device="cuda", dtype=torch.float64)
    gx, gy = px.repeat(H)[:, None], py.repeat_interleave(W)[:, None]
    ud, vd, rd = u.detach(), v.detach(), rad[order]
    inside = ((torch.floor(gx / tile_w) >= torch.floor((ud - rd) / tile_w)) &
              (torch.floor(gx / tile_w) <= torch.floor((ud + rd) / tile_w)) &
              (torch.floor(gy / tile_h) >= torch.floor((vd - rd) / tile_h)) &
              (torch.floor(gy / tile_h) <= torch.floor((vd + rd) / tile_h)))
    dx, dy = gx + 0.5 - u, gy + 0.5 - v
    a, b, c, dt = A[order], B[order], C[order], det[order]
    alpha = leaves["opacities"][order] * torch.exp(-0.5 * (c * dx * dx - 2 * b * dx * dy + a * dy * dy) / dt)
    alpha = torch.where(inside, alpha.clamp(max=float(np.float32(0.99))), torch.zeros_like(alpha))
    alpha = torch.where(alpha >= float(np.float32(1 / 255)), alpha, torch.zeros_like(alpha))
    log_T = torch.cumsum(torch.log1p(-alpha), 1)
    alpha = torch.where(torch.exp(log_T.detach()) >= float(np.float32(1e-4)), alpha, torch.zeros_like(alpha))
    before = torch.exp(log_T - torch.log1p(-alpha))
    w = torch.where(alpha > 0, alpha * before, torch.zeros_like(alpha))
    img = (w @ colour[order]).T.reshape(3, H, W)
    T = torch.exp(torch.log1p(-alpha).sum(1)).reshape(H, W)
    if dimg is None:
        return img.detach(), T.detach(), None, None
    img.backward(dimg.double())
    mean2d = torch.zeros(mu.shape[0], 2, dtype=torch.float64, device="cuda")
    mean2d[order] = splat_uv.grad
    return img.detach(), T.detach(), {k: t.grad for k, t in leaves.items()}, mean2d


def _exact_loss(s):
    x, y = s.img.double().requires_grad_(), s.target.double()
    w = torch.exp(-((torch.arange(11, device="cuda", dtype=torch.float64) - 5) ** 2) / (2 * 1.5 ** 2))
    w = w / w.sum()

    def window(a):
        # sums of shifted images: the two passes of the separable window, zero outside the image
        p = torch.nn.functional.pad(a, (5, 5))
        a = sum(w[k] * p[..., k:k + a.shape[-1]] for k in range(11))
        p = torch.nn.functional.pad(a, (0, 0, 5, 5))
        return sum(w[k] * p[..., k:k + a.shape[-2], :] for k in range(11))

    mx, my = window(x), window(y)
    sxx, syy, sxy = window(x * x) - mx * mx, window(y * y) - my * my, window(x * y) - mx * my
    c1, c2 = 0.01 ** 2, 0.03 ** 2
    ssim = ((2 * mx * my + c1) * (2 * sxy + c2) / ((mx * mx + my * my + c1) * (sxx + syy + c2))).mean()
    l1 = (x - y).abs().mean()
    loss = 0.8 * l1 + 0.2 * (1 - ssim)
    loss.backward()
    return dict(loss=torch.stack([loss, l1, ssim]).detach(), grad=x.grad)


def _exact_refine(s):
    """The decisions in 32 bits, as documented (thresholds rounded once); the values in 64."""
    p, m, v, accum, count, radius = s.inputs
    n = count.shape[0]
    f32 = lambda a: torch.tensor(np.float32(a), device="cuda")      # noqa: E731
    lim = np.float32(0.005).astype(np.float64)
    logit = f32(math.log(lim / (1 - lim)))
    big = p["log_scales"].max(1).values
    prune = ((p["logit_opacities"] < logit) | (big > f32(math.log(np.float32(0.1 * 3.0)))) | (radius > 20.0))
    dens = ~prune & (count > 0) & (accum / count > f32(0.0002))
    split = dens & (big > f32(math.log(np.float32(0.01 * 3.0))))
    copies = torch.where(prune, 0, torch.where(dens, 2, 1))
    src = torch.repeat_interleave(torch.arange(n, device="cuda"), copies)
    first = torch.cumsum(copies, 0) - copies
    child = torch.arange(src.shape[0], device="cuda") - first[src]
    normals = torch.randn((n, 2, 3), dtype=torch.float32, device="cuda", generator=s.gen.manual_seed(s.seed)).double()
    out = {k: t.double()[src] for k, t in p.items()}
    sp = split[src]
    R = _rotations(torch.nn.functional.normalize(out["quats"], dim=1))
    step = torch.einsum("nij,nj->ni", R, torch.exp(out["log_scales"]) * normals[src, child])
    out["means"] = torch.where(sp[:, None], out["means"] + step, out["means"])
    out["log_scales"] = torch.where(sp[:, None], out["log_scales"] - math.log(np.float32(1.6)), out["log_scales"])
    keep = ((child == 0) & ~sp).double()
    moments = {k: [t.double()[src] * keep.view(-1, *([1] * (t.dim() - 1))) for t in (m[k], v[k])] for k in PARAMS}
    return dict(rows=None, params=out, moments=moments, scales=torch.exp(out["log_scales"]),
                opacities=torch.sigmoid(out["logit_opacities"]))
