"""Performance cases of the framework's main paths.

Each case is one call (or the few calls a program always makes together) that a
user of the framework makes over and over: a training step, an evaluation
render, the depth order, the loss, the backward, a densification, the freeze
predictor, a step of several scenes. Inputs are drawn on the GPU from a seed
with the distributions of the synthetic workloads (``synth.py``): Gaussians in
a cube (the tiny workload) or on a sphere / plane / box mix (all others),
cameras on a hemisphere, textured targets with sensor noise.

``exact`` evaluates the same outputs in float64 with plain torch: every
(Gaussian, pixel) pair is listed, ordered by (pixel, depth) and composited with
segmented sums, and the parameter gradient comes from autograd through the
float64 projection.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2504_06716_gb300 import autograd, batch, lib, pipeline, synth
from paper_2504_06716_gb300.predictor import FreezePredictor
from paper_2504_06716_gb300.schedule import GStaConfig, GStaController

ALPHA_MIN, ALPHA_MAX, T_MIN, ZNEAR, DILATION = 1.0 / 255.0, 0.99, 1e-4, 0.2, 0.3
EXTENT = 4.4
ADAM_STEP = 5000  # optimiser steps taken before the timed one: the moments are warm
BATCH_VIEWS = 10  # cameras of a scene of the batch: every 8th held out, groups of 4 views


# ---------------------------------------------------------------- the cases


def listed():
    return [
        # the tiny workload's training step (2,000 Gaussians, 128x128: predictor training runs it
        # thousands of times): launches and latency
        dict(name="step-tiny", kind="step", n=2000, width=128, height=128, tile=16, ppt=0, batch=0, frozen=0.0,
             densify=False),
        # a step of a small scene early in the freezing window, library-default launch shapes
        dict(name="step-120k", kind="step", n=120_000, width=800, height=800, tile=16, ppt=0, batch=0, frozen=0.5,
             densify=False),
        # the benchmark's step: 1M Gaussians, GSta's freeze map (95% asleep), both statistics
        # windows, the autotuner's 8-pixel tiles and launch shapes
        dict(name="step-gsta-1m", kind="step", n=1_000_000, width=1237, height=822, tile=8, ppt=2, batch=64,
             frozen=0.95, densify=True),
        # the same step of plain 3DGS (and of GSta before its window opens): nothing asleep
        dict(name="step-plain-1m", kind="step", n=1_000_000, width=1237, height=822, tile=8, ppt=2, batch=64,
             frozen=0.0, densify=True),
        # evaluation render of the stress workload (PSNR checks, held-out views, viewers)
        dict(name="render-3m-1080p", kind="render", n=3_000_000, width=1920, height=1080, tile=16),
        # backward of one view (rasteriser and projection) of a mid-size scene
        dict(name="backward-400k", kind="backward", n=400_000, width=800, height=800, tile=16, ppt=0, batch=0,
             frozen=0.5),
        # projection and per-tile depth order on a ragged image, 8-pixel tiles
        dict(name="order-250k", kind="order", n=250_003, width=1001, height=667, tile=8),
        # the Eq. 3 loss and its gradient on one training image
        dict(name="loss-1237x822", kind="loss", width=1237, height=822),
        # the autograd API: render, loss, gradient of the parameters
        dict(name="autograd-100k", kind="autograd", n=100_000, width=512, height=512, tile=16),
        # adaptive densification of the benchmark's set (every 100 iterations)
        dict(name="densify-1m", kind="densify", n=1_000_000),
        # the learned freeze predictor over the stress workload's Gaussians: features and inference
        dict(name="predict-3m", kind="predict", n=3_000_000),
        # one graph-replayed step of three scenes of uneven size, four views each
        dict(name="batch-3-scenes", kind="batch", n=250_000, width=800, height=800, tile=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, n, w_max=1237, h_max=822):
    """An image for n Gaussians: at least a pixel for every eight of them, as late in a progressive schedule."""
    w, h = _log_int(rng, 96, w_max), _log_int(rng, 96, h_max)
    grow = max(1.0, math.sqrt(n / (8.0 * w * h)))
    return dict(width=min(w_max, int(w * grow) + 1), height=min(h_max, int(h * grow) + 1))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "render", "backward", "order", "loss", "autograd", "densify", "predict",
                       "batch"])
    tile = rng.choice([8, 16, 32])
    ppt = rng.choice([0, 1, 2])
    shape = dict(ppt=ppt, batch=rng.choice([32, 64, 128, 256]) if ppt else 0)
    frozen = round(rng.choice([0.0, rng.uniform(0.1, 0.99)]), 3)
    if kind == "step":
        n = _log_int(rng, 1500, 1_000_000)
        return dict(kind=kind, n=n, tile=tile, frozen=frozen, densify=rng.random() < 0.5, **shape, **_size(rng, n))
    if kind == "render":
        n = _log_int(rng, 2000, 3_000_000)
        return dict(kind=kind, n=n, tile=tile, **_size(rng, n, 1920, 1080))
    if kind == "backward":
        n = _log_int(rng, 2000, 1_000_000)
        return dict(kind=kind, n=n, tile=tile, frozen=frozen, **shape, **_size(rng, n))
    if kind == "order":
        n = _log_int(rng, 1000, 3_000_000)
        return dict(kind=kind, n=n, tile=tile, **_size(rng, n))
    if kind == "loss":
        return dict(kind=kind, width=_log_int(rng, 11, 1920), height=_log_int(rng, 11, 1080))
    if kind == "autograd":
        n = _log_int(rng, 2000, 500_000)
        return dict(kind=kind, n=n, tile=16, **_size(rng, n))
    if kind in ("densify", "predict"):
        return dict(kind=kind, n=_log_int(rng, 2000, 1_000_000 if kind == "densify" else 3_000_000))
    side = _log_int(rng, 200, 800)
    return dict(kind=kind, n=_log_int(rng, 20_000, 250_000), width=side, height=side, tile=rng.choice([8, 16]))


# ---------------------------------------------------------------- inputs


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _rand(g, *shape):
    return torch.rand(shape, generator=g, device="cuda")


def _randn(g, *shape):
    return torch.randn(shape, generator=g, device="cuda")


def _surface_points(g, n):
    """Points on a unit sphere, the plane y = -1.2 over [-4, 4]^2 and 20 boxes on it, about by area."""
    which = _rand(g, n)
    v = _randn(g, n, 3)
    pts = v / v.norm(dim=1, keepdim=True)
    plane = torch.stack([_rand(g, n) * 8 - 4, torch.full((n,), -1.2, device="cuda"), _rand(g, n) * 8 - 4], 1)
    pts = torch.where((which > 0.14)[:, None], plane, pts)
    bg = np.random.Generator(np.random.PCG64(12345))
    centre = torch.tensor(bg.uniform(-3, 3, (20, 2)), dtype=torch.float32, device="cuda")
    size = torch.tensor(bg.uniform(0.1, 0.6, (20, 3)), dtype=torch.float32, device="cuda")
    k = (_rand(g, n) * 20).long().clamp_(max=19)
    u = _rand(g, n, 3)
    axis = (_rand(g, n) * 3).long().clamp_(max=2)
    u.scatter_(1, axis[:, None], (u.gather(1, axis[:, None]) > 0.5).float())
    s = size[k]
    box = torch.stack([centre[k, 0] + (u[:, 0] - 0.5) * s[:, 0], -1.2 + u[:, 1] * s[:, 1],
                       centre[k, 1] + (u[:, 2] - 0.5) * s[:, 2]], 1)
    return torch.where((which > 0.86)[:, None], box, pts)


def _params(case, seed, n=None):
    """Parameter rows [n, 64]: the tiny workload's cube or the surface mix."""
    n = n or case["n"]
    g = _gen(seed)
    cube = n <= 3000
    p = torch.zeros((n, 64), device="cuda")
    if cube:
        p[:, 0:3] = _rand(g, n, 3) * 2 - 1
        p[:, 3:6] = _randn(g, n, 3) * 0.3 - 3.5
    else:
        p[:, 0:3] = _surface_points(g, n) + _randn(g, n, 3) * 0.01
        p[:, 3:6] = _randn(g, n, 3) * 0.5 - 4.5
    q = _randn(g, n, 4)
    p[:, 6:10] = q / q.norm(dim=1, keepdim=True)
    p[:, 10] = _rand(g, n) * 4 - 2
    p[:, 11:14] = _rand(g, n, 3)
    p[:, 14:59] = _randn(g, n, 45) * 0.05
    return p


def _camera(case, seed):
    """One of 24 cameras of the hemisphere rig (the circle for the tiny cube)."""
    if case["n"] <= 3000:
        return synth.circle_cameras(8, 4.0, case["width"], case["height"])[seed % 8]
    return synth.hemisphere_cameras(24, 4.0, case["width"], case["height"])[seed % 24]


def _image(h, w, seed, noise=0.03):
    """A textured image in [0, 1] with sensor noise, [3, h, w]."""
    g = _gen(1000 + seed)
    y = torch.arange(h, device="cuda", dtype=torch.float32)[:, None]
    x = torch.arange(w, device="cuda", dtype=torch.float32)[None, :]
    out = torch.zeros((3, h, w), device="cuda")
    prm = _rand(g, 3, 6, 4).cpu().numpy()
    for c in range(3):
        for a, wl, ang, ph in prm[c]:
            k = 2 * math.pi / (8 + 120 * float(wl))
            t = 2 * math.pi * float(ang)
            out[c] += (0.2 + float(a)) * torch.sin(k * (math.cos(t) * x + math.sin(t) * y) + 6.28 * float(ph))
    out = out / 6 + 0.5
    return (out + _randn(g, 3, h, w) * noise).clamp_(0, 1)


def _moments(n, seed):
    """Adam moments of a set in training: m and v of gradients around 1e-6."""
    g = _gen(2000 + seed)
    s = 1e-6 * torch.exp(_randn(g, n, 64))
    m = 0.3 * s * _randn(g, n, 64)
    s[:, 59:] = 0
    m[:, 59:] = 0
    return m, s * s


def _frozen(case, seed):
    return (_rand(_gen(3000 + seed), case["n"]) < case["frozen"]).to(torch.uint8)


def _lrs():
    # rates of a finished schedule (the exponential decay's end, applied to every group), so that the
    # scene stays the scene it is however many steps are taken on it
    return [r / 100.0 for r in pipeline.default_lrs(EXTENT)]


def _model(case, seed, trainable=True):
    n = case["n"]
    m = pipeline.Model(np.zeros((n, 59), np.float32), trainable=trainable)
    m.P.copy_(_params(case, seed))
    if trainable:
        if case.get("densify"):
            m.enable_densify()
        mm, vv = _moments(n, seed)
        m.m.copy_(mm)
        m.v.copy_(vv)
        m.step_count = ADAM_STEP
        m.frozen.copy_(_frozen(case, seed))
        m.freeze_update(0.0, 0.0, 3)  # the unfrozen list of that map
        if case["ppt"]:
            m.fwd_cfg = m.bwd_cfg = lib.raster_config(case["ppt"], case["batch"])
    cam = lib.camera(_camera(case, seed), tile=case["tile"])
    # for the lists alone: buffers of one size whatever the seed
    capacity = 24 * n + 400_000 if case["kind"] == "order" else m.measure_capacity([cam])
    return m, m.make_view(cam, capacity, trainable=trainable)


def _densify_inputs(case, seed):
    n, g = case["n"], _gen(4000 + seed)
    cnt = torch.randint(0, 100, (n,), generator=g, device="cuda", dtype=torch.int32)
    acc_xyz = cnt * 1.2e-4 * torch.exp(0.6 * _randn(g, n))  # about 15% of the averages above 2e-4
    acc_rgb = cnt * 1e-6 * torch.exp(_randn(g, n))
    radius = torch.randint(0, 40, (n,), generator=g, device="cuda", dtype=torch.int32)
    m, v = _moments(n, seed)
    frozen = (_rand(g, n) < 0.5).to(torch.uint8)
    return dict(cnt=cnt, acc_xyz=acc_xyz, acc_rgb=acc_rgb, radius=radius, m=m, v=v, frozen=frozen,
                z=_randn(g, n, 2, 3), P=_params(case, seed))


def _densify_params():
    f = lambda x: float(np.float32(x))  # noqa: E731
    return lib.GsDensifyParams(f(2e-4), f(1e-6), 0, f(math.log(0.01 * EXTENT)), f(math.log(0.005 / 0.995)), 1,
                               2**31 - 1, f(math.log(0.1 * EXTENT)), f(math.log(1.6)))


def _predict_inputs(case, seed):
    n, g = case["n"], _gen(5000 + seed)
    cnt = torch.randint(0, 60, (n,), generator=g, device="cuda", dtype=torch.int32)
    ax, ar = cnt * 3e-5 * torch.exp(_randn(g, n)), cnt * 1e-4 * torch.exp(_randn(g, n))
    state = torch.zeros((n, 12), device="cuda")
    state[:, 0:4] = 3e-5 * torch.exp(_randn(g, n, 4))
    state[:, 4:8] = 1e-4 * torch.exp(_randn(g, n, 4))
    state[:, 8], state[:, 9] = state[:, 0], state[:, 4]
    state[:, 10] = torch.randint(0, 4000, (n,), generator=g, device="cuda").float()
    state[:, 11] = torch.randint(0, 12, (n,), generator=g, device="cuda").float()
    return dict(cnt=cnt, ax=ax, ar=ar, state=state, P=_params(case, seed), k=4000, K=30000, ex=2.1e-5, er=7e-5)


def _batch_sizes(case):
    n = case["n"]
    return [n // 5, n // 2, n]  # 50K, 125K and 250K in the listed case


def _batch_rows(case, seed, i, n):
    return _params(case, 10 * seed + i, n), *_moments(n, 10 * seed + i)


def _batch_trainer(case, seed):
    cams = synth.hemisphere_cameras(BATCH_VIEWS, 4.0, case["width"], case["height"])
    train, test, subset = synth.split_views(BATCH_VIEWS, 0.1, 2)
    sizes = _batch_sizes(case)
    scenes = []
    for i, n in enumerate(sizes):
        init = _params(case, 10 * seed + i, n)[:, :59].cpu().numpy()
        scenes.append(synth.Scene(init, init[:1000], cams, train, test, subset))
    bt = batch.BatchTrainer(scenes, GStaConfig(), tile=case["tile"], fwd=(2, 64), bwd=(2, 64))
    by_size = sorted(bt.scenes, key=lambda s: s.n)
    for i, s in enumerate(by_size):
        for v, t in s.targets.items():
            t.copy_(_image(case["height"], case["width"], 100 * seed + 10 * i + v))
    for _ in range(bt.n_groups):  # captures the graph of each view group
        bt.step("graph")
    torch.cuda.synchronize()
    for i, s in enumerate(by_size):  # then the drawn state, as after loading a checkpoint
        P, m, v = _batch_rows(case, seed, i, s.n)
        s.model.P.copy_(P)
        s.model.m.copy_(m)
        s.model.v.copy_(v)
        s.step_dev.fill_(ADAM_STEP)
        s.lr_host = _lrs()
        s.lr_dev.copy_(torch.tensor(s.lr_host))
        s.ctrl = GStaController(s.cfg, s.lr_host[0])
        for t in (s.model.acc_xyz, s.model.acc_rgb, s.model.cnt):
            t.zero_()
    return bt, by_size


def _batch_group(i):
    """The four views of group 0 of the scene of size rank i (seeded permutation of the training views)."""
    train, _, _ = synth.split_views(BATCH_VIEWS, 0.1, 2)
    return [train[j] for j in np.random.default_rng(100 + i).permutation(len(train))][:4]


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("step", "backward"):
        m, view = _model(case, seed)
        st = dict(kind=kind, m=m, view=view, gt=_image(case["height"], case["width"], seed), lrs=_lrs())
        if kind == "backward":
            m.rasterize(view)
            m.loss(view, st["gt"])
        return st
    if kind == "render":
        m, view = _model(case, seed, trainable=False)
        return dict(kind=kind, m=m, view=view)
    if kind == "order":
        m, view = _model(case, seed, trainable=False)
        return dict(kind=kind, m=m, view=view)
    if kind == "loss":
        h, w = case["height"], case["width"]
        gt = _image(h, w, seed)
        img = (gt + 0.1 * (_image(h, w, seed + 50) - 0.5)).contiguous()
        return dict(kind=kind, h=h, w=w, gt=gt, img=img, dl=torch.zeros_like(img),
                    loss=torch.zeros(1, device="cuda"),
                    ws=torch.zeros(lib.gs_loss_workspace_bytes(h, w), dtype=torch.uint8, device="cuda"))
    if kind == "autograd":
        return dict(kind=kind, P=_params(case, seed).requires_grad_(True),
                    cam=lib.camera(_camera(case, seed), tile=case["tile"]),
                    gt=_image(case["height"], case["width"], seed))
    if kind == "densify":
        st, n = _densify_inputs(case, seed), case["n"]
        cap = int(1.5 * n) + 1024
        z = lambda *s, dt=torch.float32: torch.zeros(s, dtype=dt, device="cuda")  # noqa: E731
        st.update(kind=kind, n=n, cap=cap, prm=_densify_params(), counts=z(4, dt=torch.int64),
                  ws=z(lib.gs_densify_workspace_bytes(n), dt=torch.uint8), P2=z(cap, 64), m2=z(cap, 64), v2=z(cap, 64),
                  fr2=z(cap, dt=torch.uint8), ax2=z(cap), ar2=z(cap), cnt2=z(cap, dt=torch.int32))
        st["stats"] = lib.grad_stats(st["acc_xyz"], st["acc_rgb"], st["cnt"], st["radius"])
        st["carry"] = [lib.densify_carry(st[a], st[b])
                       for a, b in (("acc_xyz", "ax2"), ("acc_rgb", "ar2"), ("cnt", "cnt2"))]
        return st
    if kind == "predict":
        st, n = _predict_inputs(case, seed), case["n"]
        st.update(kind=kind, n=n, pred=FreezePredictor(seed=seed), p=torch.zeros(n, device="cuda"),
                  X=torch.zeros((n, 16), dtype=torch.bfloat16, device="cuda"))
        return st
    bt, by_size = _batch_trainer(case, seed)
    return dict(kind=kind, bt=bt, scenes=by_size)


# ---------------------------------------------------------------- one pass


def run(st):
    kind = st["kind"]
    if kind == "step":
        m, v = st["m"], st["view"]
        m.train_step(v, st["gt"], st["lrs"])
        return dict(loss=v.loss, image=v.image, G=m.G, P=m.P, m=m.m, v=m.v, acc_xyz=m.acc_xyz)
    if kind == "render":
        m, v = st["m"], st["view"]
        m.rasterize(v)
        return dict(image=v.image, t_final=v.t_final, n_last=v.n_last)
    if kind == "backward":
        m, v = st["m"], st["view"]
        m.backward(v)
        return dict(G=m.G, acc_xyz=m.acc_xyz, acc_rgb=m.acc_rgb, cnt=m.cnt)
    if kind == "order":
        m, v = st["m"], st["view"]
        lib.gs_project(m.P, m.n, m.sh_degree, v.cam, m.splats)
        lib.gs_sort(m.splats, m.n, v.cam, v.sort_ws, v.capacity, v.vals, v.ranges, v.count)
        # the records' last two words are integers
        return dict(splats=m.splats[:, :10], radius_tiles=m.splats.view(torch.int32)[:, 10:], vals=v.vals,
                    ranges=v.ranges, count=v.count)
    if kind == "loss":
        lib.gs_loss(st["img"], st["gt"], st["h"], st["w"], 0.2, st["ws"], st["loss"], st["dl"])
        return dict(loss=st["loss"], dl=st["dl"])
    if kind == "autograd":
        P = st["P"]
        P.grad = None
        image = autograd.rasterize(P, st["cam"])
        loss = autograd.ssim_l1_loss(image, st["gt"])
        loss.backward()
        return dict(loss=loss, image=image, grad=P.grad)
    if kind == "densify":
        lib.gs_densify_plan(st["n"], st["P"], st["stats"], st["prm"], st["ws"], st["counts"])
        lib.gs_densify_apply(st["n"], st["P"], st["m"], st["v"], st["frozen"], st["carry"], st["prm"], st["z"],
                             st["ws"], st["cap"], st["P2"], st["m2"], st["v2"], st["fr2"])
        return dict(counts=st["counts"], P=st["P2"], m=st["m2"], v=st["v2"], frozen=st["fr2"], acc_xyz=st["ax2"],
                    acc_rgb=st["ar2"], cnt=st["cnt2"])
    if kind == "predict":
        lib.gs_pred_features(st["n"], st["P"], st["ax"], st["ar"], st["cnt"], st["state"], st["k"], st["K"], st["ex"],
                             st["er"], st["X"])
        st["pred"].predict(st["X"], st["p"])
        return dict(X=st["X"], p=st["p"])
    st["bt"].step("graph")
    return [dict(loss=[s.view.loss for s in sc.slots], image=[s.view.image for s in sc.slots], G=sc.model.G,
                 P=sc.model.P, m=sc.model.m, v=sc.model.v) for sc in st["scenes"]]


# ---------------------------------------------------------------- the least work


def work(case):
    """Inputs read once and outputs written once. Pixel pairs: a splat of the
    surface mix covers about pi * 9 * (its squared pixel radius) pixels, and
    front-to-back compositing ends a ray after some tens of them."""
    kind = case["kind"]
    n = case.get("n", 0)
    hw = case.get("width", 0) * case.get("height", 0)
    vis = 0.6 * n
    r2 = (0.011 * case.get("width", 0) / (2 * math.tan(math.pi / 6)) / 4) ** 2 + 0.3
    pairs = min(vis * 28 * r2, 120.0 * hw)
    project = 48 * n + 192 * vis + 48 * vis
    fwd = pairs * 20.0
    active = n * (1 - case.get("frozen", 0.0))
    bwd = pairs * (20.0 + 30.0 * (active / n if n else 0))
    row = 59 * 4
    if kind == "step":
        # P read; image and target; G written, P, m and v read and written for the unfrozen
        return dict(bytes=project - 48 * vis + 24 * hw + active * (row + 5 * row), flops=fwd + bwd + 3 * 440 * hw)
    if kind == "render":
        return dict(bytes=project - 48 * vis + 20 * hw, flops=fwd)
    if kind == "backward":
        return dict(bytes=48 * vis + 20 * hw + active * (row * 2 + 24), flops=bwd)
    if kind == "order":
        return dict(bytes=project + 4 * vis * max(1.0, 28 * r2 / case["tile"] ** 2), flops=300.0 * n)
    if kind == "loss":
        return dict(bytes=36 * hw, flops=3 * 440.0 * hw)
    if kind == "autograd":
        return dict(bytes=project - 48 * vis + 24 * hw + n * row, flops=fwd + pairs * 50.0 + 3 * 440 * hw)
    if kind == "densify":
        return dict(bytes=n * (3 * 256 + 17) * 2.0, flops=40.0 * n)
    if kind == "predict":
        return dict(bytes=n * (48 + 48 + 12 + 32 + 4), flops=n * 2.0 * (16 * 64 + 64 * 64 + 64))
    total = sum(_batch_sizes(case))
    per = 4 * (fwd + pairs * 50.0 + 3 * 440 * hw)
    return dict(bytes=4 * (240 * total + 3 * 24 * hw) + total * 6 * row, flops=per * (total / n))


# ---------------------------------------------------------------- float64


class _Cam:
    """A camera's numbers as the library gets them (float32), in float64."""

    def __init__(self, c, tile):
        f = lambda a: torch.tensor(np.asarray(np.asarray(a, np.float32), np.float64), device="cuda")  # noqa: E731
        self.W, self.H, self.tile = c.width, c.height, tile
        self.fx, self.fy, self.cx, self.cy = (float(np.float32(x)) for x in (c.fx, c.fy, c.cx, c.cy))
        self.R, self.t, self.pos = f(c.R), f(c.t), f(c.campos)
        self.near, self.dil = float(np.float32(ZNEAR)), float(np.float32(DILATION))


def _sh_colour(k, d):
    """max(0, sum_c k_c Y_c(d) + 1/2), the real SH basis of degree 3 with Condon-Shortley phase."""
    x, y, z = d.unbind(1)
    pi = math.pi
    xx, yy, zz = x * x, y * y, z * z
    a1, a2, a3 = math.sqrt(3 / (4 * pi)), math.sqrt(15 / (4 * pi)), math.sqrt(35 / (32 * pi))
    b3, c3 = math.sqrt(105 / (4 * pi)), math.sqrt(21 / (32 * pi))
    Y = [torch.full_like(x, 0.5 / math.sqrt(pi)), -a1 * y, a1 * z, -a1 * x, a2 * x * y, -a2 * y * z,
         math.sqrt(5 / (16 * pi)) * (3 * zz - 1), -a2 * x * z, 0.5 * a2 * (xx - yy), -a3 * y * (3 * xx - yy),
         b3 * x * y * z, -c3 * y * (5 * zz - 1), math.sqrt(7 / (16 * pi)) * z * (5 * zz - 3), -c3 * x * (5 * zz - 1),
         0.5 * b3 * z * (xx - yy), -a3 * x * (xx - 3 * yy)]
    return (torch.einsum("nc,ncr->nr", torch.stack(Y, 1), k) + 0.5).clamp(min=0)


def _project64(P, cam):
    """Eq. 1 for the Gaussians of one view: those it sees (indices) and, differentiable in P, their
    2-D means, conics, opacities, colours; the pixel rectangles of their tiles; depths."""
    with torch.no_grad():
        front = torch.nonzero((P[:, :3] @ cam.R[2] + cam.t[2]) > cam.near).flatten()
    p = P[front]
    c = p[:, :3] @ cam.R.T + cam.t
    z = c[:, 2]
    q = p[:, 6:10] / p[:, 6:10].norm(dim=1, keepdim=True)
    w, x, y, zq = q.unbind(1)
    R = torch.stack([1 - 2 * (y * y + zq * zq), 2 * (x * y - w * zq), 2 * (x * zq + w * y),
                     2 * (x * y + w * zq), 1 - 2 * (x * x + zq * zq), 2 * (y * zq - w * x),
                     2 * (x * zq - w * y), 2 * (y * zq + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    M = R * p[:, 3:6].exp()[:, None, :]
    lim = (1.3 * 0.5 * cam.W / cam.fx, 1.3 * 0.5 * cam.H / cam.fy)
    u, v = (c[:, 0] / z).clamp(-lim[0], lim[0]), (c[:, 1] / z).clamp(-lim[1], lim[1])
    T0 = (cam.fx / z)[:, None] * cam.R[0] - (cam.fx * u / z)[:, None] * cam.R[2]
    T1 = (cam.fy / z)[:, None] * cam.R[1] - (cam.fy * v / z)[:, None] * cam.R[2]
    U0, U1 = torch.einsum("ni,nij->nj", T0, M), torch.einsum("ni,nij->nj", T1, M)
    A, B, C = (U0 * U0).sum(1) + cam.dil, (U0 * U1).sum(1), (U1 * U1).sum(1) + cam.dil
    det = A * C - B * B
    mean = torch.stack([cam.fx * c[:, 0] / z + cam.cx, cam.fy * c[:, 1] / z + cam.cy], 1)
    conic = torch.stack([C / det, -B / det, A / det], 1)
    d = p[:, :3] - cam.pos
    rgb = _sh_colour(p[:, 11:59].view(-1, 16, 3), d / d.norm(dim=1, keepdim=True))
    op = torch.sigmoid(p[:, 10])
    with torch.no_grad():
        rad = torch.ceil(3 * torch.sqrt(0.5 * (A + C) + torch.sqrt((0.5 * (A - C)) ** 2 + B * B)))
        t, n_t = cam.tile, torch.tensor([-(-cam.W // cam.tile), -(-cam.H // cam.tile)], device="cuda")
        lo = torch.floor((mean - rad[:, None]) / t).clamp(min=0).long()
        hi = torch.minimum(torch.floor((mean + rad[:, None]) / t).long() + 1, n_t)
        seen = (hi > lo).all(1) & (det > 0)
        size = torch.tensor([cam.W, cam.H], device="cuda")
        # the pixels of its tiles where alpha can reach 1/255: a box around the ellipse
        tau = 2 * torch.log((255 * op).clamp(min=1.0))
        half = torch.sqrt(tau[:, None] * torch.stack([A, C], 1)) + 1
        a = torch.maximum(lo * t, torch.ceil(mean - half).long())
        b = torch.minimum(torch.minimum(hi * t, size), torch.floor(mean + half).long() + 1)
    k = torch.nonzero(seen).flatten()
    return dict(idx=front[k], mean=mean[k], conic=conic[k], op=op[k], rgb=rgb[k], lo=a[k], hi=b[k], depth=z[k].detach())


def _pairs(s, cam, y0, y1):
    """Blended (splat, pixel) pairs of the rows y0 <= y < y1, ordered by pixel then depth:
    (splat, pixel, dx, dy, alpha, T in front, cap not reached, first pair of the pixel)."""
    n = s["idx"].numel()
    lo, hi = s["lo"].clone(), s["hi"].clone()
    lo[:, 1].clamp_(min=y0)
    hi[:, 1].clamp_(max=y1)
    wh = (hi - lo).clamp(min=0)
    cnt = wh[:, 0] * wh[:, 1]
    start = torch.cumsum(cnt, 0) - cnt
    i = torch.repeat_interleave(torch.arange(n, device="cuda"), cnt)
    o = torch.arange(i.numel(), device="cuda") - start[i]
    px, py = lo[i, 0] + o % wh[i, 0], lo[i, 1] + torch.div(o, wh[i, 0], rounding_mode="floor")
    mean, con, op = s["mean"].detach(), s["conic"].detach(), s["op"].detach()
    dx, dy = mean[i, 0] - px, mean[i, 1] - py
    power = -0.5 * (con[i, 0] * dx * dx + con[i, 2] * dy * dy) - con[i, 1] * dx * dy
    oG = op[i] * torch.exp(power)
    keep = (power <= 0) & (oG >= ALPHA_MIN)
    i, px, py, dx, dy, oG = (t[keep] for t in (i, px, py, dx, dy, oG))
    rank = torch.empty(n, dtype=torch.int64, device="cuda")
    rank[torch.argsort(s["depth"], stable=True)] = torch.arange(n, device="cuda")
    pix = py * cam.W + px
    order = torch.argsort(pix * max(n, 1) + rank[i])
    i, pix, dx, dy, oG = (t[order] for t in (i, pix, dx, dy, oG))
    alpha = oG.clamp(max=ALPHA_MAX)
    ln = torch.log1p(-alpha)
    cs = torch.cumsum(ln, 0) - ln  # in front of each pair, over all pixels
    _, counts = torch.unique_consecutive(pix, return_counts=True)
    first = torch.repeat_interleave(torch.cumsum(counts, 0) - counts, counts)
    T = torch.exp(cs - cs[first])
    live = T * (1 - alpha) >= T_MIN
    i, pix, dx, dy, alpha, T, oG = (t[live] for t in (i, pix, dx, dy, alpha, T, oG))
    return i, pix, dx, dy, alpha, T, oG <= ALPHA_MAX


def _bands(cam, n):
    rows = max(8, int(cam.H * min(1.0, 200_000 / max(n, 1)) ** 0.5))
    return [(y, min(cam.H, y + rows)) for y in range(0, cam.H, rows)]


def _render64(s, cam):
    img = torch.zeros((3, cam.H * cam.W), dtype=torch.float64, device="cuda")
    lnT = torch.zeros(cam.H * cam.W, dtype=torch.float64, device="cuda")
    rgb = s["rgb"].detach()
    for y0, y1 in _bands(cam, s["idx"].numel()):
        i, pix, _, _, al, T, _ = _pairs(s, cam, y0, y1)
        for c in range(3):
            img[c].index_add_(0, pix, al * T * rgb[i, c])
        lnT.index_add_(0, pix, torch.log1p(-al))
    return img.view(3, cam.H, cam.W), torch.exp(lnT).view(cam.H, cam.W)


def _grad64(P, s, cam, dl, frozen):
    """dL/dP [n, 64] (zero rows where frozen) and |dL/dmean2d| in device units, |dL/dk_0|."""
    n = s["idx"].numel()
    g = torch.zeros((n, 9), dtype=torch.float64, device="cuda")
    dl = dl.reshape(3, -1)
    con, rgb, op = s["conic"].detach(), s["rgb"].detach(), s["op"].detach()
    for y0, y1 in _bands(cam, n):
        i, pix, dx, dy, al, T, free = _pairs(s, cam, y0, y1)
        w = al * T
        dcc = sum(dl[c, pix] * rgb[i, c] for c in range(3))
        cs = torch.cumsum(dcc * w, 0)
        _, counts = torch.unique_consecutive(pix, return_counts=True)
        last = torch.repeat_interleave(torch.cumsum(counts, 0) - 1, counts)
        behind = cs[last] - cs  # black background
        dA = T * dcc - behind / (1 - al)
        dp = torch.where(free, dA * al, torch.zeros_like(dA))
        a, b, c_ = con[i, 0], con[i, 1], con[i, 2]
        cols = [-(a * dx + b * dy) * dp, -(b * dx + c_ * dy) * dp, -0.5 * dx * dx * dp, -dx * dy * dp,
                -0.5 * dy * dy * dp, dp / op[i]] + [w * dl[c, pix] for c in range(3)]
        for k, v in enumerate(cols):
            g[:, k].index_add_(0, i, v)
    if frozen is not None:
        g[frozen[s["idx"]] != 0] = 0
    out = torch.cat([s["mean"], s["conic"], s["op"][:, None], s["rgb"]], 1)
    (grad,) = torch.autograd.grad((out * g).sum(), P)
    nx = torch.zeros(P.shape[0], dtype=torch.float64, device="cuda")
    nx[s["idx"]] = torch.sqrt((g[:, 0] * 0.5 * cam.W) ** 2 + (g[:, 1] * 0.5 * cam.H) ** 2)
    return grad, nx, grad[:, 11:14].norm(dim=1)


def _loss64(img, gt):
    """Eq. 3 and its gradient."""
    img = img.detach().double().requires_grad_(True)
    gt = gt.double()
    w = torch.tensor([math.exp(-(k - 5) ** 2 / 4.5) for k in range(11)], dtype=torch.float64, device="cuda")
    w = w / w.sum()

    def win(x):
        x = F.conv2d(x[:, None], w.view(1, 1, 1, 11), padding=(0, 5))
        return F.conv2d(x, w.view(1, 1, 11, 1), padding=(5, 0))[:, 0]

    mx, my = win(img), win(gt)
    vx, vy, cxy = win(img * img) - mx * mx, win(gt * gt) - my * my, win(img * gt) - mx * my
    ssim = ((2 * mx * my + 1e-4) * (2 * cxy + 9e-4)) / ((mx * mx + my * my + 1e-4) * (vx + vy + 9e-4))
    lam = float(np.float32(0.2))
    loss = (1 - lam) * (img - gt).abs().mean() + lam * (1 - ssim.mean())
    (dl,) = torch.autograd.grad(loss, img)
    return loss.detach().view(1), dl


def _adam64(P, G, m, v, frozen, step):
    b1, b2 = float(np.float32(0.9)), float(np.float32(0.999))
    lr = torch.zeros(64, dtype=torch.float64, device="cuda")
    for (a, b), r in zip(((0, 3), (3, 6), (6, 10), (10, 11), (11, 14), (14, 59)), _lrs()):
        lr[a:b] = float(np.float32(r))
    m2, v2 = b1 * m + (1 - b1) * G, b2 * v + (1 - b2) * G * G
    P2 = P - lr * (m2 / (1 - b1**step)) / (torch.sqrt(v2 / (1 - b2**step)) + 1e-15)
    if frozen is not None:
        f = (frozen != 0)[:, None]
        P2, m2, v2 = torch.where(f, P, P2), torch.where(f, m, m2), torch.where(f, v, v2)
    return P2, m2, v2


def _view64(P, cam, gt, frozen):
    s = _project64(P, cam)
    img, _ = _render64(s, cam)
    loss, dl = _loss64(img, gt)
    return loss, img, *_grad64(P, s, cam, dl, frozen)


def _densify64(case, seed):
    st, prm = _densify_inputs(case, seed), _densify_params()
    n, cap = case["n"], int(1.5 * case["n"]) + 1024
    P, cnt = st["P"], st["cnt"]
    avg = torch.where(cnt > 0, st["acc_xyz"] / cnt.clamp(min=1).float(), torch.zeros_like(st["acc_xyz"]))
    cand = (cnt > 0) & (avg >= prm.eps_xyz)
    smax = P[:, 3:6].amax(1)
    clone = cand & (smax <= prm.log_clone_max)
    split = cand & ~clone
    low, big = P[:, 10] < prm.logit_min_opacity, smax > prm.log_max_world
    keep = ~split & ~low & ~big
    kid = split & ~low & ~(smax - prm.log_split_div > prm.log_max_world)
    P64 = P.double()
    q = P64[:, 6:10] / P64[:, 6:10].norm(dim=1, keepdim=True)
    rank = torch.cumsum(split.long(), 0) - 1
    kids = torch.nonzero(kid).flatten().repeat_interleave(2)
    z = st["z"].double().view(-1, 3)[2 * rank[kids] + torch.arange(kids.numel(), device="cuda") % 2]
    w, v = q[kids, 0:1], q[kids, 1:4]
    sz = P64[kids, 3:6].exp() * z
    t = 2 * torch.linalg.cross(v, sz)
    child = P64[kids].clone()
    child[:, 0:3] += sz + w * t + torch.linalg.cross(v, t)
    child[:, 3:6] -= float(np.float32(prm.log_split_div))
    rows = torch.cat([P64[keep], P64[clone & ~low & ~big], child])
    k = int(keep.sum())

    def out(x):
        o = torch.zeros((cap,) + tuple(x.shape[1:]), dtype=torch.float64, device="cuda")
        o[: x.shape[0]] = x
        return o

    return dict(counts=None, P=out(rows), m=out(st["m"][keep].double()), v=out(st["v"][keep].double()), frozen=None,
                acc_xyz=out(st["acc_xyz"][keep].double()), acc_rgb=out(st["acc_rgb"][keep].double()), cnt=None) if k else None


def _predict64(case, seed):
    st = _predict_inputs(case, seed)
    pred = FreezePredictor(seed=seed).params  # the weights are inputs
    f = lambda x: x.double()  # noqa: E731
    ex, er = float(np.float32(st["ex"])), float(np.float32(st["er"]))
    ratio = lambda v, e: torch.log10(v.clamp(min=1e-30) / e).clamp(-8, 8)  # noqa: E731
    s, P, cnt = f(st["state"]), f(st["P"]), f(st["cnt"])
    ax, ar = (torch.where(cnt > 0, f(st[k]) / cnt.clamp(min=1), torch.zeros_like(cnt)) for k in ("ax", "ar"))
    X = torch.cat([ratio(s[:, 0:4], ex), ratio(s[:, 4:8], er), torch.sigmoid(P[:, 10:11]),
                   P[:, 3:6].amax(1, keepdim=True), P[:, 3:6].amin(1, keepdim=True), torch.log1p(s[:, 10:11]),
                   torch.full_like(s[:, :1], st["k"] / st["K"]), ratio(ax, ex)[:, None], ratio(ar, er)[:, None],
                   s[:, 11:12].clamp(max=8) / 8], 1)
    bf = lambda t: t.float().to(torch.bfloat16).double()  # noqa: E731
    W1, b1, W2 = bf(pred[0:1024]).view(16, 64), f(pred[1024:1088]), bf(pred[1088:5184]).view(64, 64)
    b2, W3, b3 = f(pred[5184:5248]), bf(pred[5248:5312]), f(pred[5312:5313])
    h1 = bf((bf(X) @ W1 + b1).clamp(min=0))
    return dict(X=X, p=torch.sigmoid((h1 @ W2 + b2).clamp(min=0) @ W3 + b3))


def exact(case, seed):
    kind = case["kind"]
    if kind == "loss":
        st = prepare(case, seed)
        loss, dl = _loss64(st["img"], st["gt"])
        return dict(loss=loss, dl=dl)
    if kind == "densify":
        return _densify64(case, seed)
    if kind == "predict":
        return _predict64(case, seed)
    if kind == "batch":
        cams = synth.hemisphere_cameras(BATCH_VIEWS, 4.0, case["width"], case["height"])
        out = []
        for i, n in enumerate(_batch_sizes(case)):
            P, m, v = (t.double() for t in _batch_rows(case, seed, i, n))
            P.requires_grad_(True)
            G, losses, images = 0, [], []
            for vw in _batch_group(i):
                gt = _image(case["height"], case["width"], 100 * seed + 10 * i + vw)
                loss, img, g, _, _ = _view64(P, _Cam(cams[vw], case["tile"]), gt, None)
                G = G + g
                losses.append(loss)
                images.append(img)
            P2, m2, v2 = _adam64(P.detach(), G, m, v, None, ADAM_STEP + 1)
            out.append(dict(loss=losses, image=images, G=G, P=P2, m=m2, v=v2))
        return out
    cam = _Cam(_camera(case, seed), case["tile"])
    P = _params(case, seed).double()
    if kind in ("render", "order"):
        s = _project64(P, cam)
        if kind == "render":
            img, T = _render64(s, cam)
            return dict(image=img, t_final=T, n_last=None)
        rec = torch.zeros((case["n"], 10), dtype=torch.float64, device="cuda")
        rec[s["idx"]] = torch.cat([s["mean"], s["conic"], s["op"][:, None], s["rgb"], s["depth"][:, None]], 1)
        return dict(splats=rec, radius_tiles=None, vals=None, ranges=None, count=None)
    P.requires_grad_(True)
    frozen = _frozen(case, seed) if kind != "autograd" else None
    loss, img, G, nx, nr = _view64(P, cam, _image(case["height"], case["width"], seed), frozen)
    if kind == "autograd":
        return dict(loss=loss[0], image=img, grad=G)
    if kind == "backward":
        return dict(G=G, acc_xyz=nx, acc_rgb=nr, cnt=None)
    m, v = (t.double() for t in _moments(case["n"], seed))
    P2, m2, v2 = _adam64(P.detach(), G, m, v, frozen, ADAM_STEP + 1)
    return dict(loss=loss, image=img, G=G, P=P2, m=m2, v=v2, acc_xyz=nx)
