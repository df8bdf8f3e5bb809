"""Timed cases of the library's public entry points, with 64-bit references.

`listed()` names the cases, `draw(rng)` gives further ones of the same ranges,
`prepare(case, seed)` makes what a user's program holds before the call (seeded
inputs on the GPU, the workspace, a captured graph), `run(state)` is one pass
and `exact(case, seed)` its outputs in plain 64-bit torch.  `work(case)` is the
traffic and arithmetic a pass cannot do without.

The kinds of work, each a thing a program does with this library:

  render     forward-only render of one or several cameras into a forward-only
             workspace: a viewer's frame, a serving request, a batch of views
  autograd   the differentiable render and its backward through torch autograd:
             a small scene inside somebody else's training loop
  step       one single-view training step as a captured graph: one binning for
             the culled training render and the importance walk, loss, compact
             backward, deferred Adam, the importance selection on a second stream
  batch      one multi-view training step (train.TrainStep, captured, deferred
             Adam) with the views and targets of the next batch uploaded first
  dense      the plain training step of one view, eager: forward, loss, dense
             gradients, dense Adam
  loss       the photometric loss and its image gradient alone
  importance the scoring sweep over a set of views (s, c^rad, c^vis, Cull matrix)
  simplify   Pass 2 of the simplification: the mass cut and the compaction of the
             whole model (parameters, moments, levels)
  densify    one density-control step (clone, split, remove) of the whole model

Scenes follow the recipes of synth (the plain scene in front of one camera, the
2 km city with aerial cameras), drawn with torch on the GPU from the seed.
Learning rates are those late in training (a hundredth of the start's), so a
state can be stepped many times and still hold the same kind of scene.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2605_13794_gb300 import binding as B
from paper_2605_13794_gb300 import model as M
from paper_2605_13794_gb300 import synth
from paper_2605_13794_gb300.train import TrainStep

DEV = "cuda"
PARAMS = ("mean", "log_scale", "quat", "opacity_logit", "sh")
LOD = dict(lod_d0=1600.0, lod_Lmax=5)
LAMBDA, BETA = 0.2, 10.0
LR = [1.6e-4, 5e-5, 1e-5, 2.5e-4, 2.5e-5]  # mean, log-scale, quaternion, opacity, SH
MIXED = ((640, 480), (1280, 720), (1920, 1080), (2560, 1440), (3840, 2160))
POOL = 4  # batches of views a multi-view training loop cycles through


# ---- cases ---------------------------------------------------------------------------


def listed():
    return [
        # the smallest call: 10k Gaussians, one 256x256 camera, forward and backward
        dict(name="autograd_plain10k_256", kind="autograd", scene="plain", n=10_000, width=256, height=256),
        # small training: two views of an odd size, where launches and their gaps count
        dict(name="batch_plain20k_2x251x187", kind="batch", scene="plain", n=20_000, views=2, width=251, height=187),
        # a frame of a small scene at 720p
        dict(name="render_city200k_720p", kind="render", scene="city", n=200_000, views=1, width=1280, height=720,
             tile_w=16, tile_h=16),
        # a frame of the resident 5M city at 1080p: the render latency a viewer sees
        dict(name="render_city5M_1080p", kind="render", scene="city", n=5_000_000, views=1, width=1920, height=1080,
             tile_w=16, tile_h=16),
        # a batch of cameras of mixed resolution in one launch sequence, at the tile shape the autotuner takes
        dict(name="render_city4M_24mixed", kind="render", scene="city", n=4_000_000, views=24, width=0, height=0,
             tile_w=32, tile_h=16),
        # the single-view training step on the 5M city at 1080p
        dict(name="step_city5M_1080p", kind="step", scene="city", n=5_000_000, width=1920, height=1080),
        # the multi-view training step: eight views of 1600x1200 per step, views cycling through a pool
        dict(name="batch_city8M_8x1600x1200", kind="batch", scene="city", n=8_000_000, views=8, width=1600,
             height=1200),
        # the plain per-view path on an odd-sized image
        dict(name="dense_city1M_1277x719", kind="dense", scene="city", n=1_000_003, width=1277, height=719),
        # the loss of a batch of two odd-sized images
        dict(name="loss_2x1201x1599", kind="loss", views=2, width=1599, height=1201),
        # one chunk of the scoring sweep over the training views
        dict(name="importance_city3M_8x1080p", kind="importance", scene="city", n=3_000_000, views=8, width=1920,
             height=1080),
        # the scheduled simplification of a 3M model
        dict(name="simplify_3M", kind="simplify", n=3_000_001),
        # one density-control step of a 1.5M model
        dict(name="densify_1500k", kind="densify", n=1_500_000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["autograd", "batch", "render", "render", "render", "step", "dense", "loss", "importance",
                       "simplify", "densify"])
    tw, th = rng.choice([(16, 16), (16, 16), (16, 16), (32, 16), (32, 8), (16, 8)])
    size = dict(width=_log_int(rng, 200, 1920), height=_log_int(rng, 150, 1200))
    if kind == "autograd":
        return dict(kind=kind, scene="plain", n=_log_int(rng, 2_000, 40_000), width=rng.randint(96, 400),
                    height=rng.randint(96, 400))
    if kind == "batch":
        if rng.random() < 0.4:
            return dict(kind=kind, scene="plain", n=_log_int(rng, 5_000, 40_000), views=rng.randint(1, 4),
                        width=rng.randint(96, 400), height=rng.randint(96, 400))
        return dict(kind=kind, scene="city", n=_log_int(rng, 100_000, 6_000_000), views=rng.randint(2, 8), **size)
    if kind == "render":
        views = rng.choice([1, 1, 2, 5, 12])
        if views > 1:
            return dict(kind=kind, scene="city", n=_log_int(rng, 100_000, 4_000_000), views=views, width=0, height=0,
                        tile_w=tw, tile_h=th)
        return dict(kind=kind, scene="city", n=_log_int(rng, 20_000, 8_000_000), views=1,
                    width=_log_int(rng, 320, 3840), height=_log_int(rng, 240, 2160), tile_w=tw, tile_h=th)
    if kind in ("step", "dense"):
        return dict(kind=kind, scene="city", n=_log_int(rng, 100_000, 5_000_000 if kind == "step" else 2_000_000),
                    **size)
    if kind == "loss":
        return dict(kind=kind, views=rng.randint(1, 4), **size)
    if kind == "importance":
        return dict(kind=kind, scene="city", n=_log_int(rng, 50_000, 3_000_000), views=rng.randint(1, 8), **size)
    return dict(kind=kind, n=_log_int(rng, 20_000, 3_000_000 if kind == "simplify" else 1_500_000))


# ---- inputs: seeded, the same for the library and for the reference -------------------


def _gen(seed, salt):
    return torch.Generator(device=DEV).manual_seed(1_000_003 * int(seed) + salt)


def _rand(gen, *shape, lo=0.0, hi=1.0):
    return torch.rand(*shape, generator=gen, device=DEV) * (hi - lo) + lo


def _randn(gen, *shape, sigma=1.0):
    return torch.randn(*shape, generator=gen, device=DEV) * sigma


def _quats(gen, n):
    q = _randn(gen, n, 4)
    return (q / q.norm(dim=1, keepdim=True)).contiguous()


def _sh(gen, n):
    sh = _randn(gen, n, 16, 3, sigma=0.2)
    sh[:, 0] += 0.5
    return sh


def _plain_scene(n, seed):
    gen = _gen(seed, 11)
    mean = torch.stack([_rand(gen, n, lo=-1, hi=1), _rand(gen, n, lo=-1, hi=1), _rand(gen, n, lo=2, hi=6)], 1)
    log_scale = _rand(gen, n, 3, lo=math.log(1e-3), hi=math.log(5e-2))
    return B.GaussianTensors(mean.contiguous(), log_scale, _quats(gen, n), _randn(gen, n), _sh(gen, n),
                             torch.zeros(n, dtype=torch.uint8, device=DEV))


def _city_scene(n, seed, half=1000.0, boxes=200):
    """Ground plane (60 %) and building faces (40 %) over 2 km x 2 km, as synth.city_scene."""
    host = np.random.default_rng(1_000_003 * int(seed) + 13)
    bc, bs = host.uniform(-0.9 * half, 0.9 * half, (boxes, 2)), host.uniform(20.0, 120.0, (boxes, 2))
    bh = host.uniform(10.0, 80.0, boxes)
    area = np.stack([bs[:, 1] * bh, bs[:, 1] * bh, bs[:, 0] * bh, bs[:, 0] * bh, bs[:, 0] * bs[:, 1]], 1).ravel()
    cum = torch.from_numpy(np.cumsum(area / area.sum()).astype(np.float32)).to(DEV)
    bc, bs, bh = (torch.from_numpy(a.astype(np.float32)).to(DEV) for a in (bc, bs, bh))
    gen = _gen(seed, 17)
    ng = int(round(0.6 * n))
    nb = n - ng
    mean = torch.empty(n, 3, device=DEV)
    mean[:ng, :2] = _rand(gen, ng, 2, lo=-half, hi=half)
    mean[:ng, 2] = _randn(gen, ng, sigma=0.5)
    pick = torch.searchsorted(cum, _rand(gen, nb)).clamp_(max=5 * boxes - 1)
    b, face = pick // 5, pick % 5
    u, u2, w = _rand(gen, nb, lo=-0.5, hi=0.5), _rand(gen, nb, lo=-0.5, hi=0.5), _rand(gen, nb)
    fx = torch.where(face == 0, torch.full_like(u, -0.5), torch.where(face == 1, torch.full_like(u, 0.5), u))
    fy = torch.where(face == 2, torch.full_like(u, -0.5),
                     torch.where(face == 3, torch.full_like(u, 0.5), torch.where(face == 4, u2, u)))
    mean[ng:, 0] = bc[b, 0] + fx * bs[b, 0]
    mean[ng:, 1] = bc[b, 1] + fy * bs[b, 1]
    mean[ng:, 2] = torch.where(face == 4, bh[b], w * bh[b])
    log_scale = _randn(gen, n, 3) + math.log(0.3)
    lod = torch.round(torch.log2(2.4 / log_scale.exp().mean(1))).clamp_(0, 5).to(torch.uint8)
    return B.GaussianTensors(mean, log_scale, _quats(gen, n), _randn(gen, n), _sh(gen, n), lod)


def _scene(case, seed):
    return (_plain_scene if case["scene"] == "plain" else _city_scene)(case["n"], seed)


def _cameras(case, seed, batch=0):
    V, W, H = case.get("views", 1), case["width"], case["height"]
    rng = random.Random(1_000_003 * int(seed) + 19 + batch)
    if case["scene"] == "plain":
        f = 300.0 * max(W, H) / 256.0
        cams = [synth.plain_camera(W, H, f)]
        for _ in range(1, V):
            pos = (rng.uniform(-0.6, 0.6), rng.uniform(-0.6, 0.6), rng.uniform(-0.6, 0.2))
            cams.append(synth.look_at_camera(pos, (0.0, 0.0, 4.0), (0.0, -1.0, 0.0), W, H, 50.0))
        return cams
    if W == 0:  # mixed resolutions (in turn) and distances
        return [synth.mixed_cameras(1, rng.randrange(1 << 30), sizes=(MIXED[k % len(MIXED)],))[0] for k in range(V)]
    return [synth.aerial_camera(rng.randrange(1 << 30), width=W, height=H) for _ in range(V)]


def _target(V, H, W, seed, batch=0):
    """Photograph-like targets: a smooth field with noise, in [0, 1]."""
    gen = _gen(seed, 23 + batch)
    coarse = _rand(gen, V, 3, max(2, H // 24), max(2, W // 24))
    img = torch.nn.functional.interpolate(coarse, size=(H, W), mode="bilinear", align_corners=False)
    return (0.85 * img + 0.15 * _rand(gen, V, 3, H, W)).contiguous()


def _cull_column(n, seed):
    """A Cull column with a third of the Gaussians culled."""
    words = (n + 31) // 32
    bits = _rand(_gen(seed, 29), words * 32) < 1.0 / 3.0
    bits[n:] = False
    weights = (torch.ones(32, dtype=torch.int64, device=DEV) << torch.arange(32, device=DEV))
    packed = (bits.view(words, 32).to(torch.int64) * weights).sum(1)
    packed = torch.where(packed >= 1 << 31, packed - (1 << 32), packed)
    return packed.to(torch.int32), bits[:n]


def _params(case, **over):
    d = dict(tile_w=case.get("tile_w", 16), tile_h=case.get("tile_h", 16))
    if case["scene"] == "city":
        d.update(lod_enable=True, **LOD)
    if case["kind"] in ("render", "autograd"):
        d.update(bg=(0.1, 0.2, 0.3))
    d.update(over)
    return B.RenderParams(**d)


def _pixels(cams):
    return sum(c.width * c.height for c in cams)


def _capacity(g, batches, params, headroom):
    """Records and instances the views need (the largest batch), with headroom for training."""
    tw, th = params.tile_w, params.tile_h
    cams = max(batches, key=_pixels)
    probe = B.Workspace(max_gaussians=g.n, max_records=min(g.n * len(cams), 1 << 26), max_instances=1 << 26,
                        max_tiles=sum(B.tiles_of(c, tw, th) for c in cams), max_pixels=_pixels(cams),
                        max_cameras=len(cams), forward_only=True)
    rec = inst = 0
    for b in batches:
        probe.preprocess(g, b, params)
        probe.bin_sort()
        c = probe.counts()
        rec, inst = max(rec, c["records_needed"]), max(inst, c["instances_needed"])
    probe.close()
    return dict(max_records=min(g.n * len(cams), int(rec * headroom) + 8192),
                max_instances=min((1 << 30) - 1, int(inst * headroom) + 65536))


def _workspace(g, cams, params, cap, **kw):
    return B.Workspace(max_gaussians=g.n, max_tiles=sum(B.tiles_of(c, params.tile_w, params.tile_h) for c in cams),
                       max_pixels=_pixels(cams), max_cameras=len(cams), **cap, **kw)


_warmed = []


def _warm_up():
    """One small eager training step per process, so that every kernel is loaded before a capture."""
    if _warmed:
        return
    case = dict(kind="batch", scene="plain", n=2000, views=1, width=64, height=48)
    g, cams = _scene(case, 0), _cameras(case, 0)
    ts = TrainStep(g, cams, _target(1, 48, 64, 0), _params(case), LR, LAMBDA, BETA, lazy=True)
    words = torch.zeros((g.n + 31) // 32, dtype=torch.int32, device=DEV)
    ts.run()
    ts.ws.preprocess(g, cams, _params(case, cull_enable=B.GS_CULL_MARK), words)
    ts.ws.bin_sort()
    ts.ws.render_fwd_importance(ts.rgb)
    ts.ws.importance(cull_out=words)
    ts.run()
    ts.flush()
    ts.ws.sync_status()
    ts.ws.close()
    _warmed.append(True)


# ---- prepare and run, by kind ------------------------------------------------------------


def _prepare_render(case, seed):
    g, cams, params = _scene(case, seed), _cameras(case, seed), _params(case)
    ws = _workspace(g, cams, params, _capacity(g, [cams], params, 1.3), forward_only=True)
    P = _pixels(cams)
    return dict(ws=ws, g=g, cams=cams, params=params, rgb=torch.empty(3 * P, device=DEV),
                T=torch.empty(P, device=DEV))


def _run_render(s):
    s["ws"].preprocess(s["g"], s["cams"], s["params"])
    s["ws"].bin_sort()
    s["ws"].render_fwd(s["rgb"], s["T"])
    return dict(rgb=s["rgb"], T=s["T"])


def _prepare_autograd(case, seed):
    g, cams, params = _scene(case, seed), _cameras(case, seed), _params(case)
    ws = _workspace(g, cams, params, dict(max_records=g.n, max_instances=64 * g.n))
    dL = _randn(_gen(seed, 31), 3 * _pixels(cams))
    for p in g.params():
        p.requires_grad_(True)
    return dict(ws=ws, g=g, cams=cams, params=params, dL=dL)


def _run_autograd(s):
    rgb, T = B.render(s["ws"], s["g"], s["cams"], s["params"])
    grads = torch.autograd.grad(rgb, s["g"].params(), s["dL"])
    return dict(rgb=rgb.detach(), T=T, grads=dict(zip(PARAMS, grads)))


def _prepare_step(case, seed):
    _warm_up()
    g, cams = _scene(case, seed), _cameras(case, seed)
    params = _params(case, cull_enable=B.GS_CULL_MARK)
    ws = _workspace(g, cams, params, _capacity(g, [cams], _params(case), 1.5))
    H, W, n, P = case["height"], case["width"], g.n, _pixels(cams)
    z = lambda *shape, dtype=torch.float32: torch.zeros(*shape, dtype=dtype, device=DEV)
    s = dict(ws=ws, g=g, cams=cams, params=params, m=g.zeros_like(), v=g.zeros_like(), last=z(n, dtype=torch.int32),
             drift=z(2, n), rgb=z(3 * P), T=z(P), dL=z(3 * P), loss=z(1), reg=z(1), s=z(n),
             crad=z(n, dtype=torch.int32), cvis=z(n, dtype=torch.int32), cull=_cull_column(n, seed)[0],
             cull_next=z((n + 31) // 32, dtype=torch.int32), target=_target(1, H, W, seed))
    ws.adam_lazy_enable(s["m"], s["v"], s["last"], s["drift"], max_steps=1 << 16)
    ws.upload_cameras(cams, params)
    main, side = torch.cuda.Stream(), torch.cuda.Stream()
    s["graph"] = graph = B.Graph()
    torch.cuda.synchronize()
    with graph.capture(main):
        ws.preprocess_uploaded(g, params, s["cull"])
        ws.bin_sort()
        ws.render_fwd_importance(s["rgb"], s["T"])
        side.wait_stream(main)
        ws.importance(s_accum=s["s"], crad=s["crad"], cvis=s["cvis"], cull_out=s["cull_next"], stream=side)
        ws.photometric_loss(s["rgb"].view(1, 3, H, W), s["target"], LAMBDA, s["loss"], s["dL"])
        ws.render_bwd_compact(g, s["dL"], scale_reg_beta=BETA, scale_reg_value=s["reg"])
        ws.adam_step_compact(g, s["m"], s["v"], LR, 0)
        main.wait_stream(side)
    s["streams"] = (main, side)
    return s


def _tensors(g):
    return dict(zip(PARAMS, g.params()))


def _run_step(s):
    s["graph"].launch()
    return dict(rgb=s["rgb"], T=s["T"], loss=s["loss"], reg=s["reg"], s=s["s"], crad=s["crad"], cvis=s["cvis"],
                cull=s["cull_next"], params=_tensors(s["g"]), m=_tensors(s["m"]), v=_tensors(s["v"]))


def _prepare_batch(case, seed):
    _warm_up()
    g, params = _scene(case, seed), _params(case)
    batches = [_cameras(case, seed, k) for k in range(POOL)]
    targets = [_target(case["views"], case["height"], case["width"], seed, k) for k in range(POOL)]
    ts = TrainStep(g, batches[0], targets[0], params, LR, LAMBDA, BETA, lazy=True,
                   capacity=_capacity(g, batches, params, 1.5))
    torch.cuda.synchronize()
    ts.capture()
    return dict(ts=ts, batches=batches, targets=targets, at=0)


def _run_batch(s):
    ts, k = s["ts"], s["at"]
    s["at"] = (k + 1) % POOL
    ts.set_views(s["batches"][k], s["targets"][k])
    ts.replay()
    return dict(rgb=ts.rgb, loss=ts.loss, reg=ts.reg, params=_tensors(ts.g), m=_tensors(ts.m), v=_tensors(ts.v))


def _prepare_dense(case, seed):
    g, cams, params = _scene(case, seed), _cameras(case, seed), _params(case)
    ws = _workspace(g, cams, params, _capacity(g, [cams], params, 1.5))
    P, H, W = _pixels(cams), case["height"], case["width"]
    e = lambda k: torch.zeros(k, device=DEV)
    return dict(ws=ws, g=g, cams=cams, params=params, m=g.zeros_like(), v=g.zeros_like(), grads=g.zeros_like(),
                rgb=e(3 * P), dL=e(3 * P), loss=e(1), absgrad=e(g.n), target=_target(1, H, W, seed), step=0, H=H, W=W)


def _run_dense(s):
    ws, g = s["ws"], s["g"]
    s["step"] += 1
    ws.preprocess(g, s["cams"], s["params"])
    ws.bin_sort()
    ws.render_fwd(s["rgb"])
    ws.photometric_loss(s["rgb"].view(1, 3, s["H"], s["W"]), s["target"], LAMBDA, s["loss"], s["dL"])
    ws.render_bwd(g, s["dL"], s["grads"], absgrad=s["absgrad"])
    B.adam_step([(p, gr, m, v, LR[k], 0.9, 0.999, 1e-15) for k, (p, gr, m, v) in
                 enumerate(zip(g.params(), s["grads"].params(), s["m"].params(), s["v"].params()))], step=s["step"])
    return dict(rgb=s["rgb"], loss=s["loss"], absgrad=s["absgrad"], grads=_tensors(s["grads"]), params=_tensors(g),
                m=_tensors(s["m"]), v=_tensors(s["v"]))


def _loss_inputs(case, seed):
    V, H, W = case["views"], case["height"], case["width"]
    target = _target(V, H, W, seed)
    return (target + _randn(_gen(seed, 37), V, 3, H, W, sigma=0.1)).contiguous(), target


def _prepare_loss(case, seed):
    image, target = _loss_inputs(case, seed)
    V, H, W = case["views"], case["height"], case["width"]
    ws = B.Workspace(max_gaussians=1, max_records=1, max_instances=1, max_tiles=1, max_pixels=V * H * W)
    return dict(ws=ws, image=image, target=target, loss=torch.zeros(1, device=DEV), dL=torch.empty_like(image))


def _run_loss(s):
    s["ws"].photometric_loss(s["image"], s["target"], LAMBDA, s["loss"], s["dL"])
    return dict(loss=s["loss"], dL=s["dL"])


def _prepare_importance(case, seed):
    g, cams, params = _scene(case, seed), _cameras(case, seed), _params(case)
    ws = _workspace(g, cams, params, _capacity(g, [cams], params, 1.3), forward_only=True)
    return dict(ws=ws, g=g, cams=cams, params=params)


def _run_importance(s):
    return M.importance_sweep(s["ws"], s["g"], s["cams"], s["params"])


# The quantities that decide how many rows a model pass writes (scores, opacities, scales,
# densification statistics) are one population per size, dealt to the Gaussians by the seed,
# so every seed of a case gives outputs of one size.


def _deal(n, seed):
    return torch.randperm(n, generator=_gen(seed, 39), device=DEV)


def _model(case, seed):
    """A model in mid-training: parameters, moments, levels."""
    n = case["n"]
    g, base, deal = _city_scene(n, seed), _gen(0, 40), _deal(n, seed)
    g.opacity_logit = _randn(base, n)[deal]
    g.log_scale = (_randn(base, n, 3) + math.log(0.3))[deal]
    gen = _gen(seed, 41)
    m = B.GaussianTensors(*[_randn(gen, *p.shape, sigma=1e-4) for p in g.params()], None)
    v = B.GaussianTensors(*[_rand(gen, *p.shape) * 1e-7 for p in g.params()], None)
    return B.ModelTensors(g, m, v)


def _scores(n, seed):
    """Importance scores: heavy-tailed, a fifth of the Gaussians never seen."""
    base = _gen(0, 43)
    s = torch.exp(_randn(base, n, sigma=1.5) - 3.0)
    return torch.where(_rand(base, n) < 0.2, torch.zeros_like(s), s)[_deal(n, seed)]


def _prepare_simplify(case, seed):
    n = case["n"]
    ws = B.Workspace(max_gaussians=n, max_records=1, max_instances=1, max_tiles=1, max_pixels=1, model_ops=True)
    return dict(ws=ws, model=_model(case, seed), s=_scores(n, seed))


def _rows(model):
    return dict(params=_tensors(model.g), lod=model.g.lod, m=_tensors(model.m), v=_tensors(model.v))


def _run_simplify(s):
    return _rows(M.simplify(s["ws"], s["model"], s["s"], pass_no=2))


def _densify_inputs(n, seed):
    base, deal = _gen(0, 47), _deal(n, seed)
    denom = torch.randint(0, 9, (n,), generator=base, device=DEV, dtype=torch.int32)
    crad = denom + torch.randint(0, 4, (n,), generator=base, device=DEV, dtype=torch.int32)
    cvis = (crad * _rand(base, n)).to(torch.int32)
    absgrad = denom * torch.exp(_randn(base, n) - 8.5)
    return absgrad[deal], denom[deal], cvis[deal], crad[deal]


def _prepare_densify(case, seed):
    n = case["n"]
    ws = B.Workspace(max_gaussians=n, max_records=1, max_instances=1, max_tiles=1, max_pixels=1, model_ops=True)
    return dict(ws=ws, model=_model(case, seed), stats=_densify_inputs(n, seed), seed=int(seed))


def _run_densify(s):
    return _rows(M.densify(s["ws"], s["model"], *s["stats"], seed=s["seed"], dense_scale=0.5))


_KINDS = {k: (globals()["_prepare_" + k], globals()["_run_" + k]) for k in
          ("render", "autograd", "step", "batch", "dense", "loss", "importance", "simplify", "densify")}


def prepare(case, seed):
    return dict(_KINDS[case["kind"]][0](case, seed), kind=case["kind"])


def run(state):
    return _KINDS[state["kind"]][1](state)


# ---- the work a pass cannot do without ---------------------------------------------------


def work(case):
    """Bytes: every input read once, every output written once (a render reads each Gaussian's
    mean and level and the whole rows of those in view, about a fiftieth of a city; a training
    step reads and writes the rows, moments and gradients of those; dense Adam and the model
    passes stream the whole model).  Flops: the compositing of the pairs that count (about ten
    per pixel on a city view, a hundred on the small plain scene), and the loss's two blurs."""
    kind, V = case["kind"], case.get("views", 1)
    n = case.get("n", 0)
    W, H = case.get("width", 0), case.get("height", 0)
    px = V * (W * H if W else sum(w * h for w, h in MIXED) / len(MIXED))
    if kind == "loss":
        return dict(bytes=36.0 * px, flops=3 * 2 * 11 * 2 * 8.0 * px)
    if kind in ("simplify", "densify"):
        return dict(bytes=2 * 12 * 59.0 * n, flops=10.0 * n)
    plain = case["scene"] == "plain"
    seen, pairs = (n, 100.0) if plain else (0.02 * n * min(V, 8), 10.0)
    bytes_ = 13.0 * n + 236.0 * seen + 16.0 * px
    flops = 25.0 * pairs * px + 500.0 * seen
    if kind in ("autograd", "step", "batch", "dense"):
        bytes_ += 236.0 * seen + 12.0 * px
        flops += 75.0 * pairs * px + 1500.0 * seen
    if kind in ("step", "batch", "dense"):
        bytes_ += 36.0 * px + 24 * 59.0 * (n if kind == "dense" else seen)
        flops += 1056.0 * px
    if kind == "importance":
        bytes_ += 13.0 * n
    return dict(bytes=bytes_, flops=flops)


# ---- the 64-bit reference ------------------------------------------------------------------
# The method in plain torch, FP64, written from its equations: EWA projection of the gated
# Gaussians, tile lists ordered by (depth, index), front-to-back compositing with the alpha
# and transmittance thresholds as FP32 constants, the adjoint of the compositing in closed
# form and that of the projection by autograd.

_F = lambda x: float(np.float32(x))
A_MIN, A_MAX, T_MIN, DILATION, ZNEAR, FOV_CLAMP = _F(1 / 255), _F(0.99), _F(1e-4), _F(0.3), _F(0.2), _F(1.3)
CHUNK = 1 << 25  # (tile, entry, pixel) triples per chunk


def _exact_project(p, cam, tw, th):
    """Differentiable projection of the rows of p (FP64, one camera): dict of per-row tensors."""
    t64 = lambda a: torch.as_tensor(np.asarray(a, np.float64), device=DEV)
    R, t, pos = t64(cam.R).view(3, 3), t64(cam.t), t64(cam.campos)
    fx, fy, cx, cy = (float(np.float32(x)) for x in (cam.fx, cam.fy, cam.cx, cam.cy))
    x = p["mean"] @ R.T + t
    z = x[:, 2]
    q = p["quat"] / p["quat"].norm(dim=1, keepdim=True)
    w, i, j, k = q.unbind(1)
    Q = torch.stack([1 - 2 * (j * j + k * k), 2 * (i * j - w * k), 2 * (i * k + w * j),
                     2 * (i * j + w * k), 1 - 2 * (i * i + k * k), 2 * (j * k - w * i),
                     2 * (i * k - w * j), 2 * (j * k + w * i), 1 - 2 * (i * i + j * j)], 1).view(-1, 3, 3)
    S = Q * p["log_scale"].exp()[:, None, :]
    lx, ly = FOV_CLAMP * cam.width / (2 * fx), FOV_CLAMP * cam.height / (2 * fy)
    xc, yc = (x[:, 0] / z).clamp(-lx, lx), (x[:, 1] / z).clamp(-ly, ly)
    zero = torch.zeros_like(z)
    J = torch.stack([fx / z, zero, -fx * xc / z, zero, fy / z, -fy * yc / z], 1).view(-1, 2, 3)
    V = J @ R @ S
    cov = V @ V.transpose(1, 2)
    a, b, c = cov[:, 0, 0] + DILATION, cov[:, 0, 1], cov[:, 1, 1] + DILATION
    det = a * c - b * b
    mid = 0.5 * (a + c)
    radius = torch.ceil(3 * (mid + (mid * mid - det).clamp(min=_F(0.1)).sqrt()).sqrt()).detach()
    u, v = fx * x[:, 0] / z + cx, fy * x[:, 1] / z + cy
    tx, ty = (cam.width + tw - 1) // tw, (cam.height + th - 1) // th
    edge = lambda e, size, top, one: (torch.floor(e.detach() / size) + one).clamp(0, top).long()
    rect = [edge(u - radius, tw, tx, 0), edge(v - radius, th, ty, 0), edge(u + radius, tw, tx, 1),
            edge(v + radius, th, ty, 1)]
    d = p["mean"] - pos
    d = d / d.norm(dim=1, keepdim=True)
    X, Y, Z = d.unbind(1)
    xx, yy, zz = X * X, Y * Y, Z * Z
    s = lambda num, den: math.sqrt(num / (den * math.pi))
    basis = torch.stack([
        torch.full_like(X, s(1, 4)), -s(3, 4) * Y, s(3, 4) * Z, -s(3, 4) * X,
        s(15, 4) * X * Y, -s(15, 4) * Y * Z, s(5, 16) * (2 * zz - xx - yy), -s(15, 4) * X * Z, s(15, 16) * (xx - yy),
        -s(35, 32) * Y * (3 * xx - yy), s(105, 4) * X * Y * Z, -s(21, 32) * Y * (4 * zz - xx - yy),
        s(7, 16) * Z * (2 * zz - 3 * xx - 3 * yy), -s(21, 32) * X * (4 * zz - xx - yy),
        s(105, 16) * Z * (xx - yy), -s(35, 32) * X * (xx - 3 * yy)], 1)
    rgb = ((basis[:, :, None] * p["sh"]).sum(1) + 0.5).clamp(min=0)
    return dict(u=u, v=v, A=c / det, B=-b / det, C=a / det, o=torch.sigmoid(p["opacity_logit"]), rgb=rgb, z=z,
                rect=rect, tiles=((rect[2] - rect[0]) * (rect[3] - rect[1])).detach(), ok=(det > 0) & (z > ZNEAR))


class _ExactView:
    """One camera's records, tile lists and compositing."""

    def __init__(self, g, cam, tw, th, lod, bg=(0.0, 0.0, 0.0), culled=None):
        self.cam, self.tw, self.th = cam, tw, th
        self.bg = torch.tensor([_F(b) for b in bg], dtype=torch.float64, device=DEV)
        mean = g["mean"].double()
        keep = torch.ones(len(mean), dtype=torch.bool, device=DEV)
        if lod:
            d2 = (mean - torch.as_tensor(np.asarray(cam.campos, np.float64), device=DEV)).square().sum(1)
            lv = g["lod"].long()
            limit = (LOD["lod_d0"] * 2.0 ** (0.5 - lv.double())) ** 2
            keep = (lv == 0) | ((lv <= LOD["lod_Lmax"]) & (d2 <= limit.float().double()))
        R = torch.as_tensor(np.asarray(cam.R, np.float64), device=DEV)
        keep &= mean @ R[2] + float(np.float64(cam.t[2])) > ZNEAR
        near = torch.nonzero(keep).squeeze(1)
        active = []
        for part in near.split(1 << 19):
            q = _exact_project({k: g[k][part].double() for k in PARAMS}, cam, tw, th)
            active.append(part[q["ok"] & (q["tiles"] > 0)])
        self.idx = torch.cat(active)
        self.rows = {k: g[k][self.idx].double().requires_grad_(True) for k in PARAMS}
        self.q = _exact_project(self.rows, cam, tw, th)
        q = {k: v.detach() for k, v in self.q.items() if torch.is_tensor(v)}
        self.d = q
        self.culled = culled[self.idx] if culled is not None else torch.zeros_like(self.idx, dtype=torch.bool)
        self.o = q["o"] * (~self.culled)
        # instances in (tile, depth bits, index) order
        x0, y0, x1, _ = self.q["rect"]
        n = q["tiles"]
        rec = torch.repeat_interleave(torch.arange(len(n), device=DEV), n)
        local = torch.arange(len(rec), device=DEV) - (n.cumsum(0) - n)[rec]
        w = (x1 - x0)[rec]
        self.tx, self.ty = (cam.width + tw - 1) // tw, (cam.height + th - 1) // th
        tile = (y0[rec] + local // w) * self.tx + x0[rec] + local % w
        bits = q["z"].float().view(torch.int32).long()
        order = torch.sort((tile << 32) | bits[rec], stable=True).indices
        self.list, tile = rec[order], tile[order]
        self.count = torch.bincount(tile, minlength=self.tx * self.ty)
        self.start = self.count.cumsum(0) - self.count

    def _chunks(self, opacity):
        """Tiles by list length, in chunks: (tile pixel indices, entry ids, composited terms)."""
        cam, tw, th, d = self.cam, self.tw, self.th, self.d
        order = torch.argsort(self.count, descending=True)
        length = self.count[order].tolist()
        ly, lx = torch.meshgrid(torch.arange(th, device=DEV), torch.arange(tw, device=DEV), indexing="ij")
        at = 0
        while at < len(length) and length[at] > 0:
            L = length[at]
            nt = max(1, CHUNK // (L * tw * th))
            tiles = order[at:at + nt]
            at += nt
            entry = torch.arange(L, device=DEV)
            have = entry[None] < self.count[tiles][:, None]
            rec = torch.where(have, self.list[(self.start[tiles][:, None] + entry[None]).clamp(max=len(self.list) - 1)],
                              torch.zeros_like(entry)[None])
            px = (tiles % self.tx * tw)[:, None] + lx.reshape(1, -1)
            py = (tiles // self.tx * th)[:, None] + ly.reshape(1, -1)
            inside = (px < cam.width) & (py < cam.height)
            col = lambda t: t[rec][:, :, None]
            dx, dy = px[:, None, :] + 0.5 - col(d["u"]), py[:, None, :] + 0.5 - col(d["v"])
            A, Bc, C = col(d["A"]), col(d["B"]), col(d["C"])
            G = torch.exp(-0.5 * (A * dx * dx + C * dy * dy) - Bc * dx * dy)
            raw = (opacity[rec] * have)[:, :, None] * G
            alpha = raw.clamp(max=A_MAX)
            alpha = torch.where(alpha >= A_MIN, alpha, torch.zeros_like(alpha))
            Tin = torch.cumprod(1 - alpha, 1)
            on = (alpha > 0) & (Tin >= T_MIN) & inside[:, None, :]
            alpha = torch.where(on, alpha, torch.zeros_like(alpha))
            Tin = torch.cumprod(1 - alpha, 1)
            T = torch.cat([torch.ones_like(Tin[:, :1]), Tin[:, :-1]], 1)
            yield dict(px=px, py=py, inside=inside, rec=rec, have=have, dx=dx, dy=dy, A=A, B=Bc, C=C, G=G, raw=raw,
                       alpha=alpha, on=on, T=T, T_final=Tin[:, -1])

    def image(self):
        H, W = self.cam.height, self.cam.width
        img = self.bg[:, None, None].expand(3, H, W).clone()
        T = torch.ones(H, W, dtype=torch.float64, device=DEV)
        for c in self._chunks(self.o):
            out = torch.einsum("tlp,tlc->tpc", c["alpha"] * c["T"], self.d["rgb"][c["rec"]])
            out = out + c["T_final"][:, :, None] * self.bg
            m = c["inside"]
            img[:, c["py"][m], c["px"][m]] = out[m].T
            T[c["py"][m], c["px"][m]] = c["T_final"][m]
        return img, T

    def backward(self, dL):
        """Gradients of the scene's rows of this camera for dL (3, H, W): dict by parameter, and |dL/d(u, v)|."""
        n = len(self.idx)
        g = {k: torch.zeros(n, dtype=torch.float64, device=DEV) for k in ("u", "v", "A", "B", "C", "o")}
        grgb = torch.zeros(n, 3, dtype=torch.float64, device=DEV)
        for c in self._chunks(self.o):
            m = c["inside"]
            gp = torch.zeros(*m.shape, 3, dtype=torch.float64, device=DEV)
            gp[m] = dL[:, c["py"][m], c["px"][m]].T
            rec, w = c["rec"], c["alpha"] * c["T"]
            gc = torch.einsum("tpc,tlc->tlp", gp, self.d["rgb"][rec])
            behind = (w * gc).flip(1).cumsum(1).flip(1) - w * gc + (c["T_final"] * (gp @ self.bg))[:, None, :]
            dal = torch.where(c["on"] & (c["raw"] < A_MAX), c["T"] * gc - behind / (1 - c["alpha"]),
                              torch.zeros_like(w))
            dG = dal * c["G"]
            dpow = dal * c["raw"]
            dx, dy = c["dx"], c["dy"]
            add = lambda k, t: g[k].index_add_(0, rec.reshape(-1), (t.sum(2) * c["have"]).reshape(-1))
            add("o", dG)
            add("u", dpow * (c["A"] * dx + c["B"] * dy))
            add("v", dpow * (c["C"] * dy + c["B"] * dx))
            add("A", -0.5 * dpow * dx * dx)
            add("B", -dpow * dx * dy)
            add("C", -0.5 * dpow * dy * dy)
            grgb.index_add_(0, rec.reshape(-1), (torch.einsum("tlp,tpc->tlc", w, gp) * c["have"][:, :, None])
                            .reshape(-1, 3))
        outs = [self.q[k] for k in ("u", "v", "A", "B", "C", "o", "rgb")]
        grads = torch.autograd.grad(outs, [self.rows[k] for k in PARAMS],
                                    [g["u"], g["v"], g["A"], g["B"], g["C"], g["o"], grgb])
        return dict(zip(PARAMS, grads)), torch.hypot(g["u"], g["v"])

    def importance(self):
        """w and a of each record, at its own opacity."""
        w = torch.zeros(len(self.idx), dtype=torch.float64, device=DEV)
        a = torch.zeros_like(w)
        for c in self._chunks(self.d["o"]):
            w.index_add_(0, c["rec"].reshape(-1), (c["alpha"] * c["T"]).sum(2).reshape(-1))
            a.index_add_(0, c["rec"].reshape(-1), (c["on"].sum(2) * c["have"]).double().reshape(-1))
        return w, a


def _exact_loss(image, target, lam=LAMBDA):
    """Loss and dL/dimage of a batch (V, 3, H, W), FP64."""
    x, y = image.double().requires_grad_(True), target.double()
    k = torch.exp(-(torch.arange(11, dtype=torch.float64, device=DEV) - 5) ** 2 / (2 * 1.5 ** 2))
    k = (k / k.sum()).tolist()
    H, W = x.shape[2:]

    def blur(t):
        t = torch.nn.functional.pad(t, (5, 5, 5, 5))
        t = sum(k[i] * t[..., i:i + W] for i in range(11))
        return sum(k[i] * t[..., i:i + H, :] for i in range(11))

    loss = 0.0
    for b in range(x.shape[0]):  # view by view: the memory of one
        xb, yb = x[b:b + 1], y[b:b + 1]
        mx, my = blur(xb), blur(yb)
        sx, sy, sxy = blur(xb * xb) - mx * mx, blur(yb * yb) - my * my, blur(xb * yb) - mx * my
        c1, c2 = 0.01 ** 2, 0.03 ** 2
        ssim = ((2 * mx * my + c1) * (2 * sxy + c2)) / ((mx * mx + my * my + c1) * (sx + sy + c2))
        part = ((1 - lam) * (xb - yb).abs().mean() + lam * (1 - ssim.mean())) / x.shape[0]
        part.backward()
        loss = loss + part.detach()
    return loss.reshape(1), x.grad


def _exact_adam(p, g, lr):
    """The first Adam step from zero moments: (p, m, v), FP64."""
    b1, b2 = _F(0.9), _F(0.999)
    m, v = (1 - b1) * g, (1 - b2) * g * g
    return p - lr / (1 - b1) * m / (v.sqrt() / math.sqrt(1 - b2) + 1e-15), m, v


def _detached(g):
    return dict({k: getattr(g, k).detach() for k in PARAMS}, lod=g.lod)


def _exact_train(case, seed, culled=None, dense=False, sweep=False):
    """The first training step over the case's views."""
    g = _detached(_scene(case, seed))
    n, V, H, W = case["n"], case.get("views", 1), case["height"], case["width"]
    cams, lod = _cameras(case, seed), case["scene"] == "city"
    views = [_ExactView(g, c, 16, 16, lod, culled=culled) for c in cams]
    images = [v.image() for v in views]
    rgb = torch.stack([i[0] for i in images])
    loss, dL = _exact_loss(rgb, _target(V, H, W, seed))
    grads = {k: torch.zeros(g[k].shape, dtype=torch.float64, device=DEV) for k in PARAMS}
    absgrad = torch.zeros(n, dtype=torch.float64, device=DEV)
    seen = torch.zeros(n, dtype=torch.bool, device=DEV)
    for v, d in zip(views, dL):
        gr, ab = v.backward(d)
        for k in PARAMS:
            grads[k].index_add_(0, v.idx, gr[k])
        absgrad.index_add_(0, v.idx, ab)
        seen[v.idx[~v.culled]] = True
    out = dict(rgb=rgb.reshape(-1), loss=loss)
    if not dense:
        s = g["log_scale"].double().exp()
        least = s.argmin(1)
        smin = s.gather(1, least[:, None]).squeeze(1) * seen
        nv = seen.sum().clamp(min=1)
        grads["log_scale"].scatter_add_(1, least[:, None], (BETA * smin / nv)[:, None])
        out["reg"] = (BETA * smin.sum() / nv).reshape(1)
    else:
        out["absgrad"] = absgrad
        out["grads"] = {k: grads[k] for k in PARAMS}
    if sweep:
        w, a = views[0].importance()
        out["T"] = images[0][1].reshape(-1)
        out["s"] = torch.zeros(n, dtype=torch.float64, device=DEV).index_copy_(
            0, views[0].idx, torch.where(a > 0, w / (a + _F(1e-6)), torch.zeros_like(w)))
        out.update(crad=None, cvis=None, cull=None)
    stepped = {k: _exact_adam(g[k].double(), grads[k], _F(LR[i])) for i, k in enumerate(PARAMS)}
    for j, name in enumerate(("params", "m", "v")):
        out[name] = {k: stepped[k][j] for k in PARAMS}
    return out


def _exact_render(case, seed):
    g, cams, lod = _detached(_scene(case, seed)), _cameras(case, seed), case["scene"] == "city"
    rgb, T = [], []
    for c in cams:
        i, t = _ExactView(g, c, case["tile_w"], case["tile_h"], lod, bg=(0.1, 0.2, 0.3)).image()
        rgb.append(i.reshape(-1))
        T.append(t.reshape(-1))
    return dict(rgb=torch.cat(rgb), T=torch.cat(T))


def _exact_autograd(case, seed):
    g, cam = _detached(_scene(case, seed)), _cameras(case, seed)[0]
    dL = _randn(_gen(seed, 31), 3 * cam.width * cam.height).double().view(3, cam.height, cam.width)
    view = _ExactView(g, cam, 16, 16, False, bg=(0.1, 0.2, 0.3))
    img, T = view.image()
    gr, _ = view.backward(dL)
    grads = {k: torch.zeros(g[k].shape, dtype=torch.float64, device=DEV).index_copy_(0, view.idx, gr[k])
             for k in PARAMS}
    return dict(rgb=img.reshape(-1), T=T.reshape(-1), grads=grads)


def _exact_step(case, seed):
    return _exact_train(case, seed, culled=_cull_column(case["n"], seed)[1], sweep=True)


def _exact_importance(case, seed):
    g, n = _detached(_scene(case, seed)), case["n"]
    s = torch.zeros(n, dtype=torch.float64, device=DEV)
    for c in _cameras(case, seed):
        v = _ExactView(g, c, 16, 16, True)
        w, a = v.importance()
        s.index_add_(0, v.idx, torch.where(a > 0, w / (a + _F(1e-6)), torch.zeros_like(w)))
    return dict(s=s, crad=None, cvis=None, cull=None)


def _exact_simplify(case, seed):
    s, model = _scores(case["n"], seed), _model(case, seed)
    by = torch.sort(s, descending=True, stable=True).indices
    cum = s[by].double().cumsum(0)
    first = (cum - s[by].double() < _F(0.99) * cum[-1]) & (s[by] > 0)
    rows = torch.sort(by[first]).values
    take = lambda t: {k: getattr(t, k)[rows].double() for k in PARAMS}
    return dict(params=take(model.g), lod=None, m=take(model.m), v=take(model.v))


def _exact_densify(case, seed):
    n, model = case["n"], _model(case, seed)
    absgrad, denom, cvis, crad = _densify_inputs(n, seed)
    z = torch.randn(n, 2, 3, device=DEV, generator=torch.Generator(device=DEV).manual_seed(int(seed))).double()
    g = {k: getattr(model.g, k).double() for k in PARAMS}
    # the decisions are FP32 comparisons of the stored values
    grad = torch.where(denom > 0, absgrad / denom.clamp(min=1).float(), torch.zeros_like(absgrad))
    score = grad * (cvis.float() / (crad.float() + torch.tensor(1e-6, device=DEV)))
    chosen = score >= torch.tensor(0.0002, device=DEV)
    small = model.g.log_scale.max(1).values <= float(np.float32(math.log(_F(0.5))))
    low = _F(0.005)
    removed = model.g.opacity_logit < float(np.float32(math.log(low / (1 - low))))
    split, clone = chosen & ~small & ~removed, chosen & small & ~removed
    copies = torch.where(removed, 0, torch.where(chosen, 2, 1))
    src = torch.repeat_interleave(torch.arange(n, device=DEV), copies)
    child = torch.arange(len(src), device=DEV) - (copies.cumsum(0) - copies)[src]
    out = {k: g[k][src].clone() for k in PARAMS}
    new = split[src] | (clone[src] & (child == 1))
    at = torch.nonzero(split[src]).squeeze(1)
    i = src[at]
    q = g["quat"][i] / g["quat"][i].norm(dim=1, keepdim=True)
    w, xyz = q[:, :1], q[:, 1:]
    off = g["log_scale"][i].exp() * z[i, child[at]]
    turn = 2 * torch.linalg.cross(xyz, off, dim=1)
    out["mean"][at] = g["mean"][i] + off + w * turn + torch.linalg.cross(xyz, turn, dim=1)
    out["log_scale"][at] = g["log_scale"][i] - math.log(_F(1.6))
    moment = lambda t: {k: getattr(t, k)[src].double() * (~new).view(-1, *[1] * (getattr(t, k).dim() - 1))
                        for k in PARAMS}
    return dict(params=out, lod=None, m=moment(model.m), v=moment(model.v))


_EXACT = dict(render=_exact_render, autograd=_exact_autograd, step=_exact_step, batch=_exact_train,
              dense=lambda case, seed: _exact_train(case, seed, dense=True),
              loss=lambda case, seed: dict(zip(("loss", "dL"), _exact_loss(*_loss_inputs(case, seed)))),
              importance=_exact_importance, simplify=_exact_simplify, densify=_exact_densify)


def exact(case, seed):
    return _EXACT[case["kind"]](case, seed)
