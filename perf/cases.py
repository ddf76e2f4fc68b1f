"""Performance cases of the framework: what its users run, each through a public entry point.

Kinds of work (the "kind" of a case):

  train    one training iteration of Trainer.step: render, loss (L1, or L1 + D-SSIM), backward, Adam
  render   one evaluation view of Rasterizer.render, the pair buffers grown on demand
  autograd a render and its gradient through autograd.rasterize under a loss the user wrote in torch
  batch    one captured BatchTrainer.step over several views of several scenes of uneven size
  init     Initializer.paper_init: exact kNN, neighbourhood features and the paper's seeding
  mlp      MLP.forward: the learned initializer's network over the points of one or more scenes
  fit      one minibatch step of the learned initializer's training (gradient and Adam)
  mvs      MultiViewStereo.reconstruct: depth range, reference, depth map and fused points of a target
  ba       BundleAdjuster.solve: Levenberg-Marquardt over cameras and points from a perturbed start

Scenes are the synthetic stand-ins the framework trains on: points on random spheres and squares seen
by a ring of cameras (or a uniform cloud for the smallest), drawn on the GPU from the seed alone.
exact() restates each path in 64 bits with plain torch operations.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2601_17354_gb300 import synthetic as S

DEV = "cuda"
ADAM_T = 250  # completed iterations of a trainer in mid-training (of the paper's 500)
#: root mean square of the gradient of the mean L1 loss per parameter group times the Gaussian count, measured on
#: the surface scenes: the Adam moments of a trainer in mid-training are drawn at this scale
GRAD_RMS = {"means": 10.0, "log_scales": 0.4, "quats": 0.17, "opacity_logits": 0.12, "sh": 0.25}
#: a trainer's learning rates decayed to a hundredth, as towards the end of a run: passes cost the same however many ran before
DECAY = 0.01
LR = {"means": 3.2e-4, "log_scales": 5e-3, "quats": 1e-3, "opacity_logits": 2.5e-2, "dc": 2.5e-3, "rest": 1.25e-4}
B1, B2, EPS = 0.9, 0.999, 1e-15


# ------------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------------

def _train(name, n, deg, w, h, scene="surface", tile=16, dssim=0.0):
    return {"name": name, "kind": "train", "n": n, "deg": deg, "w": w, "h": h, "scene": scene, "tile": tile,
            "dssim": dssim}


def listed():
    return [
        # the smallest training run: a thumbnail preview, 2,000 degree-0 Gaussians at 128 x 128
        _train("train_2k_128", 2000, 0, 128, 128, scene="cloud"),
        # the paper's plain loop: 100k Gaussians at 1280 x 720, one view an iteration, at the tile edge its tuner picks
        _train("train_100k_720p", 100_000, 3, 1280, 720, tile=8),
        # the headline workload: 500k Gaussians, degree 3, 1920 x 1080
        _train("train_500k_1080p", 500_000, 3, 1920, 1080),
        # L1 + D-SSIM training of a phone-sized scene at a resolution no tile divides
        _train("train_dssim_61k_1237x693", 61_003, 2, 1237, 693, dssim=0.2),
        # an evaluation render of a held-out view (PSNR of a trained model)
        {"name": "render_200k_720p", "kind": "render", "n": 200_000, "deg": 3, "w": 1280, "h": 720, "tile": 16},
        # a user's own loss on a small capture, through torch's autograd
        {"name": "autograd_30k_637x479", "kind": "autograd", "n": 30_011, "deg": 1, "w": 637, "h": 479, "tile": 16},
        # many small captures trained together in one graph
        {"name": "batch_6x4", "kind": "batch", "scenes": 6, "views": 4, "n_lo": 20_000, "n_hi": 150_000, "deg": 3,
         "tile": 16},
        # seeding one dense point cloud
        {"name": "init_200k", "kind": "init", "n": 200_000, "deg": 3},
        # the learned initializer over the points of 32 scenes
        {"name": "mlp_6400k", "kind": "mlp", "n": 6_400_000},
        # one minibatch of the learned initializer's training
        {"name": "fit_65536", "kind": "fit", "n": 65_536},
        # one keyframe's dense depth and points
        {"name": "mvs_640x360x64", "kind": "mvs", "w": 640, "h": 360, "planes": 64, "sparse": 20_000},
        # the bundle adjustment of a capture's keyframes
        {"name": "ba_32x20k", "kind": "ba", "cams": 32, "points": 20_000, "iters": 6},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["train", "train", "train", "train", "render", "autograd", "batch", "init", "mlp", "fit", "mvs",
                       "ba"])
    if kind in ("train", "render", "autograd"):
        w = _log(rng, 96, 1920)
        h = max(64, min(1080, int(w * rng.uniform(0.5, 1.0))))
        # captures hold at most about one Gaussian per four pixels (the headline workload's density)
        c = {"kind": kind, "n": _log(rng, 2000, min(500_000, max(2500, w * h // 4))), "deg": rng.randint(0, 3), "w": w,
             "h": h, "tile": rng.choice([8, 16, 16, 32])}
        if kind == "train":
            c["scene"] = "cloud" if c["n"] <= 4000 else "surface"
            c["dssim"] = rng.choice([0.0, 0.0, 0.2])
        return c
    if kind == "batch":
        lo = _log(rng, 2000, 30_000)
        return {"kind": kind, "scenes": rng.randint(2, 6), "views": rng.randint(1, 4), "n_lo": lo,
                "n_hi": _log(rng, lo, 150_000), "deg": rng.randint(0, 3), "tile": rng.choice([8, 16, 16])}
    if kind == "init":
        return {"kind": kind, "n": _log(rng, 3000, 200_000), "deg": rng.randint(0, 3)}
    if kind == "mlp":
        return {"kind": kind, "n": _log(rng, 1000, 6_400_000)}
    if kind == "fit":
        return {"kind": kind, "n": _log(rng, 1000, 65_536)}
    if kind == "mvs":
        w = rng.randint(160, 640)
        return {"kind": kind, "w": w, "h": max(90, min(360, int(w * rng.uniform(0.5, 0.75)))),
                "planes": rng.choice([32, 48, 64]), "sparse": _log(rng, 2000, 20_000)}
    return {"kind": "ba", "cams": rng.randint(8, 32), "points": _log(rng, 1000, 20_000), "iters": rng.randint(3, 6)}


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _surface_points(surf, n, g):
    """n points [3][n] on the surfaces in proportion to area."""
    dev = lambda a: torch.from_numpy(np.asarray(a, np.float32)).to(DEV)
    which = torch.multinomial(dev(surf.areas()), n, replacement=True, generator=g)
    ns = len(surf.sphere_r)
    d = torch.randn((n, 3), device=DEV, generator=g)
    d = d / d.norm(dim=1, keepdim=True)
    k = which.clamp(max=ns - 1)
    ball = dev(surf.sphere_c)[k] + dev(surf.sphere_r)[k, None] * d
    q = (which - ns).clamp(min=0)
    ab = (torch.rand((n, 2), device=DEV, generator=g) - 0.5) * dev(surf.plane_side)[q, None]
    flat = dev(surf.plane_c)[q] + ab[:, :1] * dev(surf.plane_u)[q] + ab[:, 1:] * dev(surf.plane_v)[q]
    return torch.where((which < ns)[:, None], ball, flat).t().contiguous()


def _attributes(pts, deg, g, log_scale=-4.0, logit=(1.0, 0.5)):
    """Gaussian attributes around centres [3][n]: the planar groups, by name."""
    n, K = pts.shape[1], (deg + 1) ** 2
    r = lambda *s: torch.randn(s, device=DEV, generator=g)
    sh = 0.05 * r(3, K, n)
    sh[:, 0] = (torch.rand((3, n), device=DEV, generator=g) - 0.5) * math.sqrt(4 * math.pi)
    return {"means": pts, "log_scales": log_scale + 0.3 * r(3, n), "quats": r(4, n),
            "opacity_logits": logit[0] + logit[1] * r(n), "sh": sh}


def _picture(surf, cam, g, points=400_000):
    """A photo-like [3][H][W] target: coloured surface points splatted nearest first into their pixels, smoothed."""
    pts = _surface_points(surf, points, g)
    vm = torch.from_numpy(np.asarray(cam.viewmat)).to(DEV)
    p = vm[:, :3] @ pts + vm[:, 3:]
    x = (cam.fx * p[0] / p[2] + cam.cx).floor().long()
    y = (cam.fy * p[1] / p[2] + cam.cy).floor().long()
    ok = (p[2] > 0.2) & (x >= 0) & (x < cam.width) & (y >= 0) & (y < cam.height)
    key = (p[2].view(torch.int32).long() << 20) | torch.arange(points, device=DEV)
    far = torch.full((cam.width * cam.height,), 1 << 62, device=DEV)
    far = far.scatter_reduce(0, (y * cam.width + x)[ok], key[ok], "amin")
    colour = 0.5 + 0.5 * torch.sin(6.0 * pts) * torch.cos(17.0 * pts.roll(1, 0))
    img = torch.where((far < 1 << 62)[None], colour[:, (far & 0xFFFFF).clamp(max=points - 1)], 0.0)
    img = img.view(1, 3, cam.height, cam.width)
    return torch.nn.functional.avg_pool2d(img, 5, 1, 2, count_include_pad=False)[0].contiguous()


def _view(w, h, rng):
    """One camera of the ring at the framework's field of view."""
    return S.ring_cameras(rng, 64, w, h, 1000.0 * w / 1280.0)[int(rng.integers(64))]


def _scene(case, seed):
    """(parameter groups, camera, target) of a single-view case."""
    rng, g = np.random.default_rng(seed), _gen(seed)
    if case.get("scene") == "cloud":
        pts = 2.0 * torch.rand((3, case["n"]), device=DEV, generator=g) - 1.0
        vm = np.eye(3, 4, dtype=np.float32)
        vm[2, 3] = 3.0
        f = 150.0 * case["w"] / 128.0
        cam = S.Camera(case["w"], case["h"], f, f, case["w"] / 2.0, case["h"] / 2.0, vm)
        target = torch.rand((3, case["h"], case["w"]), device=DEV, generator=g)
        return _attributes(pts, case["deg"], g, -3.0, (0.0, 1.0)), cam, target
    surf = S.random_surfaces(rng)
    cam = _view(case["w"], case["h"], rng)
    pts = _surface_points(surf, case["n"], g)
    pts += 0.01 * torch.randn(pts.shape, device=DEV, generator=g)
    return _attributes(pts, case["deg"], g), cam, _picture(surf, cam, g)


def _batch_scenes(case, seed):
    """Per scene (parameter groups, cameras, targets): counts log-uniform, three resolutions."""
    rng, g = np.random.default_rng(seed), _gen(seed)
    out, sizes = [], [(640, 480), (960, 720), (1280, 720)]
    for k in range(case["scenes"]):
        # the counts spread over the range in the same way whatever the seed, so that a pass costs the same
        u = (k + 0.5) / case["scenes"]
        n = int(round(math.exp(math.log(case["n_lo"]) * (1 - u) + math.log(case["n_hi"]) * u)))
        w, h = sizes[k % 3]
        surf = S.random_surfaces(rng)
        cams = S.ring_cameras(rng, 64, w, h, 1000.0 * w / 1280.0)
        cams = [cams[int(i)] for i in rng.integers(64, size=case["views"])]
        pts = _surface_points(surf, n, g)
        pts += 0.01 * torch.randn(pts.shape, device=DEV, generator=g)
        out.append((_attributes(pts, case["deg"], g), cams, [_picture(surf, c, g) for c in cams]))
    return out


def _moments(n, deg, seed):
    """Adam moments [rows][n] of a trainer in mid-training."""
    g = _gen(seed + 7919)
    rows = 11 + 3 * (deg + 1) ** 2
    scale = torch.empty((rows, 1), device=DEV)
    at = 0
    for name, k in (("means", 3), ("log_scales", 3), ("quats", 4), ("opacity_logits", 1), ("sh", rows - 11)):
        scale[at:at + k] = GRAD_RMS[name] / n
        at += k
    size = scale * torch.exp(0.7 * torch.randn((1, n), device=DEV, generator=g))
    m = 0.3 * size * torch.randn((rows, n), device=DEV, generator=g)
    v = size.square() * (0.5 + torch.rand((rows, n), device=DEV, generator=g))
    return m, v


def _buffer(groups, deg):
    from paper_2601_17354_gb300.rasterizer import GaussianBuffer
    buf = GaussianBuffer(groups["means"].shape[1], deg, DEV)
    for k, t in groups.items():
        getattr(buf, k).copy_(t)
    return buf


def _adam():
    from paper_2601_17354_gb300.rasterizer import AdamConfig
    return AdamConfig(lr=tuple(DECAY * LR[k] for k in ("means", "log_scales", "quats", "opacity_logits", "dc", "rest")))


def _mlp_rows(n, seed):
    """Neighbourhood features [n][16] as the network sees them, and its targets [n][8]."""
    g = _gen(seed)
    r = lambda *s: torch.randn(s, device=DEV, generator=g)
    ev = torch.rand((n, 3), device=DEV, generator=g).sort(1).values
    axes = torch.nn.functional.normalize(r(n, 3, 3), dim=2).reshape(n, 9)
    x = torch.cat([ev / ev.sum(1, keepdim=True), axes, 0.2 * r(n, 3), 11.0 + r(n, 1)], 1)
    q = torch.nn.functional.normalize(torch.cat([1 + 0.2 * r(n, 1), 0.3 * r(n, 3)], 1), dim=1)
    return x.to(torch.bfloat16), torch.cat([0.3 * r(n, 3), q, 1.0 + 0.5 * r(n, 1)], 1)


def _mvs_scene(case, seed):
    t = 4 + seed % 50
    sc = S.mvs_scene(seed, 64, case["w"], case["h"], 500.0 * case["w"] / 640.0, case["sparse"],
                     views=[t - 2, t - 1, t, t + 1, t + 2])
    return sc, t


def _ba_problem(case, seed):
    """Starting state, observations and intrinsics: every point seen by 2-12 consecutive keyframes."""
    p = S.ba_problem(seed, case["cams"], case["points"])
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
    C, n = case["cams"], case["points"]
    x = torch.einsum("cij,nj->cni", dev(p.R_gt), dev(p.P_gt)) + dev(p.t_gt)[:, None]
    uv = torch.stack([p.K[0] * x[..., 0] / x[..., 2] + p.K[2], p.K[1] * x[..., 1] / x[..., 2] + p.K[3]], -1)
    since = (torch.arange(C, device=DEV)[:, None] - dev(p.track_start)[None]) % C
    ok = (x[..., 2] > 0.2) & (uv >= 0).all(-1) & (uv[..., 0] < p.width) & (uv[..., 1] < p.height)
    ok &= since < dev(p.track_len)[None]
    ok &= ok.sum(0)[None] >= 2
    pt, cam = ok.t().nonzero(as_tuple=True)  # by point, then camera
    uv = (uv + dev(p.noise))[cam, pt].float().contiguous()
    f = lambda a: dev(np.asarray(a, np.float32))
    return f(p.R_init), f(p.t_init), f(p.P_init), cam.int(), pt.int(), uv, p.K


# ------------------------------------------------------------------------------------------------
# what a program has in hand, and one pass
# ------------------------------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        from paper_2601_17354_gb300.rasterizer import Rasterizer, Trainer
        groups, cam, target = _scene(case, seed)
        params = _buffer(groups, case["deg"])
        probe = Rasterizer(tile=case["tile"])  # the pair capacity of this view with headroom, as training loops do
        probe.render(params, cam)
        pairs = probe.status()[1]
        probe.close()
        tr = Trainer(params, Rasterizer(pair_capacity=int(1.5 * pairs) + 4096, adam=_adam(), tile=case["tile"]),
                     dssim=case["dssim"])
        m, v = _moments(case["n"], case["deg"], seed)
        tr.m.data.copy_(m)
        tr.v.data.copy_(v)
        tr.t = ADAM_T
        return {"kind": kind, "trainer": tr, "cam": cam, "target": target}
    if kind == "render":
        from paper_2601_17354_gb300.rasterizer import Rasterizer
        groups, cam, _ = _scene(case, seed)
        return {"kind": kind, "rast": Rasterizer(tile=case["tile"]), "params": _buffer(groups, case["deg"]), "cam": cam}
    if kind == "autograd":
        from paper_2601_17354_gb300.rasterizer import Rasterizer
        groups, cam, target = _scene(case, seed)
        leaves = {k: t.contiguous().requires_grad_() for k, t in groups.items()}
        return {"kind": kind, "rast": Rasterizer(tile=case["tile"]), "leaves": leaves, "cam": cam, "target": target}
    if kind == "batch":
        from paper_2601_17354_gb300.batch import BatchTrainer
        bufs, views = [], []
        for k, (groups, cams, targets) in enumerate(_batch_scenes(case, seed)):
            bufs.append(_buffer(groups, case["deg"]))
            views += [(k, c, t) for c, t in zip(cams, targets)]
        bt = BatchTrainer(bufs, views, adam=_adam(), tile=case["tile"])
        for k, b in enumerate(bufs):
            m, v = _moments(b.n, case["deg"], seed + k)
            bt.m[k].data.copy_(m)
            bt.v[k].data.copy_(v)
        bt.capture()
        return {"kind": kind, "batch": bt}
    if kind == "init":
        from paper_2601_17354_gb300.initializer import Initializer
        rng, g = np.random.default_rng(seed), _gen(seed)
        pts = _surface_points(S.random_surfaces(rng), case["n"], g)
        pts += 0.01 * torch.randn(pts.shape, device=DEV, generator=g)
        return {"kind": kind, "init": Initializer(), "points": pts, "deg": case["deg"]}
    if kind in ("mlp", "fit"):
        from paper_2601_17354_gb300.initializer import MLP, Initializer
        x, t = _mlp_rows(case["n"], seed)
        return {"kind": kind, "mlp": MLP(Initializer(), seed=seed), "x": x, "t": t}
    if kind == "mvs":
        from paper_2601_17354_gb300.mvs import MultiViewStereo
        sc, t = _mvs_scene(case, seed)
        images = [None if im is None else torch.from_numpy(im).to(DEV) for im in sc.images]
        return {"kind": kind, "mvs": MultiViewStereo(case["w"], case["h"], case["planes"]), "cams": sc.cameras,
                "images": images, "target": t, "sparse": torch.from_numpy(sc.sparse.astype(np.float32)).to(DEV)}
    from paper_2601_17354_gb300.ba import BundleAdjuster
    R, t, P, cam, pt, uv, K = _ba_problem(case, seed)
    return {"kind": kind, "ba": BundleAdjuster(case["cams"], case["points"], len(cam)), "start": (R, t, P),
            "obs": (cam, pt, uv), "K": K, "iters": case["iters"]}


def run(state):
    kind = state["kind"]
    if kind == "train":
        tr = state["trainer"]
        loss = tr.step(state["cam"], state["target"])
        return {"loss": loss, "image": tr.image, "params": tr.params.data, "m": tr.m.data, "v": tr.v.data}
    if kind == "render":
        return {"image": state["rast"].render(state["params"], state["cam"])}
    if kind == "autograd":
        from paper_2601_17354_gb300.autograd import rasterize
        p = state["leaves"]
        image = rasterize(state["rast"], state["cam"], p["means"], p["log_scales"], p["quats"], p["opacity_logits"],
                          p["sh"])
        loss = (image - state["target"]).square().mean()
        grads = torch.autograd.grad(loss, list(p.values()))
        return {"loss": loss, "image": image, "grads": dict(zip(p, grads))}
    if kind == "batch":
        bt = state["batch"]
        bt.step()
        return {"params": [b.data for b in bt.scenes], "m": [b.data for b in bt.m], "v": [b.data for b in bt.v]}
    if kind == "init":
        pi = state["init"].paper_init(state["points"], state["deg"])
        return {"params": pi.paper.data, "features": pi.features, "features_bf16": pi.features_bf16,
                "frame_q": pi.frame_q, "nb": pi.nb}
    if kind == "mlp":
        return {"y": state["mlp"].forward(state["x"])}
    if kind == "fit":
        net = state["mlp"]
        net.loss_sum.zero_()
        net.accumulate_grad(state["x"], state["t"])
        net.adam(3e-3)
        return {"loss": net.loss_sum.float(), "master": net.master, "m": net.m, "v": net.v}
    if kind == "mvs":
        ref, (lo, hi), depth, pts, pix = state["mvs"].reconstruct(state["cams"], state["images"], state["target"],
                                                                  state["sparse"])
        cloud = torch.zeros((depth.numel(), 3), device=DEV)  # organised by pixel, as viewers take a keyframe's points
        cloud[pix.long()] = pts
        return {"reference": ref, "range": [lo, hi], "depth": depth, "cloud": cloud}
    # the solve refines its arguments in place; the caller keeps the starting estimate
    R, t, P = (a.clone() for a in state["start"])
    costs, _ = state["ba"].solve(R, t, P, *state["obs"], state["K"], 0.5, 2.0, iters=state["iters"])
    # costs of a float32 state, as exact as that state
    return {"R": R, "t": t, "P": P, "costs": costs.astype(np.float32)}


def work(case):
    """Bytes: inputs read once and outputs written once.  Operations: the arithmetic of the path; for the rasterizer
    an estimate (16 per evaluated and 10 or 38 per composited entry and pixel forward or backward, at the number of
    entries a pixel of the surface scenes composites)."""
    kind = case["kind"]
    rows = lambda deg: 11 + 3 * (deg + 1) ** 2

    def entries(n, w, h):
        sigma = 1000.0 * w / 1280.0 * math.exp(-4.0) / 4.0
        return min(0.5 * n * 9 * math.pi * (sigma * sigma + 0.3), 50.0 * w * h)

    if kind in ("train", "render", "autograd"):
        n, px = case["n"], case["w"] * case["h"]
        e = entries(n, case["w"], case["h"])
        if kind == "render":
            return {"bytes": 4 * rows(case["deg"]) * n + 12 * px, "flops": 26 * e}
        if kind == "autograd":
            return {"bytes": 8 * rows(case["deg"]) * n + 24 * px, "flops": 80 * e}
        return {"bytes": 24 * rows(case["deg"]) * n + 24 * px, "flops": 80 * e}
    if kind == "batch":
        b = f = 0
        for k in range(case["scenes"]):
            u = (k + 0.5) / case["scenes"]
            n = math.exp(math.log(case["n_lo"]) * (1 - u) + math.log(case["n_hi"]) * u)
            w, h = [(640, 480), (960, 720), (1280, 720)][k % 3]
            b += 24 * rows(case["deg"]) * n + 12 * case["views"] * w * h
            f += 80 * case["views"] * entries(n, w, h)
        return {"bytes": b, "flops": f}
    if kind == "init":
        # points, 32 neighbours, fp32 and bf16 features, eigenframe and parameters; a hundred candidates a point
        n = case["n"]
        return {"bytes": n * (12 + 128 + 64 + 32 + 16 + 4 * rows(case["deg"])), "flops": n * (100 * 8 + 2000)}
    if kind == "mlp":
        return {"bytes": case["n"] * 64, "flops": case["n"] * 11264}
    if kind == "fit":
        return {"bytes": case["n"] * 64 + 6000 * 28, "flops": case["n"] * 3 * 11264}
    if kind == "mvs":
        px = case["w"] * case["h"]
        return {"bytes": px * (24 + 4 + 16) + 12 * case["sparse"], "flops": px * case["planes"] * 60}
    m = 5.5 * case["points"]
    return {"bytes": m * 16 + 24 * case["points"] + 96 * case["cams"], "flops": case["iters"] * m * 900}


# ------------------------------------------------------------------------------------------------
# 64-bit restatements
# ------------------------------------------------------------------------------------------------

def _sh_basis(d, K):
    x, y, z = d
    pi = math.pi
    c = lambda a, b: math.sqrt(a / (b * pi))
    one = torch.ones_like(x)
    b = [c(1, 4) * one, c(3, 4) * y, c(3, 4) * z, c(3, 4) * x,
         c(15, 4) * x * y, c(15, 4) * y * z, c(5, 16) * (3 * z * z - 1), c(15, 4) * x * z, c(15, 16) * (x * x - y * y),
         c(35, 32) * y * (3 * x * x - y * y), c(105, 4) * x * y * z, c(21, 32) * y * (5 * z * z - 1),
         c(7, 16) * z * (5 * z * z - 3), c(21, 32) * x * (5 * z * z - 1), c(105, 16) * z * (x * x - y * y),
         c(35, 32) * x * (x * x - 3 * y * y)]
    return torch.stack(b[:K])


def _rot(q):
    w, x, y, z = q / q.norm(dim=0)
    return [[1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)],
            [2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)],
            [2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]]


class _Raster64:
    """Render and gradient of one view in 64 bits: pinhole EWA projection, tile lists by the 3-sigma ellipse, and
    front-to-back compositing with the 0.99 / 1/255 / 1e-4 rules, differentiated by autograd."""

    CHUNK = 1 << 25  # (pixel, entry) evaluations held at a time

    def __init__(self, groups, cam, T):
        self.leaves = {k: t.detach().double().requires_grad_() for k, t in groups.items()}
        self.cam, self.T = cam, T
        self.TX, self.TY = -(-cam.width // T), -(-cam.height // T)
        self.rec = self._project()
        self._lists()

    def _project(self):
        p, cam = self.leaves, self.cam
        vm = torch.from_numpy(np.asarray(cam.viewmat, np.float64)).to(DEV)
        W, t = vm[:, :3], vm[:, 3]
        x, y, z = W @ p["means"] + t[:, None]
        self.z = z.detach()
        fx, fy = float(np.float32(cam.fx)), float(np.float32(cam.fy))
        tx, ty = x / z, y / z
        u, v = fx * tx + cam.cx, fy * ty + cam.cy
        R = _rot(p["quats"])
        s = p["log_scales"].exp()
        M = [[R[a][k] * s[k] for k in range(3)] for a in range(3)]
        Sg = [[sum(M[a][k] * M[b][k] for k in range(3)) for b in range(3)] for a in range(3)]
        lx, ly = 1.3 * 0.5 * cam.width / fx, 1.3 * 0.5 * cam.height / fy
        J = [[fx / z, -fx * tx.clamp(-lx, lx) / z], [fy / z, -fy * ty.clamp(-ly, ly) / z]]
        A = [[J[r][0] * W[r, k] + J[r][1] * W[2, k] for k in range(3)] for r in range(2)]
        q = lambda a, b: sum(A[a][m] * Sg[m][k] * A[b][k] for m in range(3) for k in range(3))
        a, b, c = q(0, 0) + 0.3, q(0, 1), q(1, 1) + 0.3
        det = a * c - b * b
        eye = -(W.t() @ t)
        d = p["means"] - eye[:, None]
        K = p["sh"].shape[1]
        rgb = (torch.einsum("ckn,kn->cn", p["sh"], _sh_basis(d / d.norm(dim=0), K)) + 0.5).clamp(min=0)
        self.ext = torch.stack([(3 * a.detach().sqrt()).ceil(), (3 * c.detach().sqrt()).ceil()])
        self.seen = (self.z > float(np.float32(cam.near))) & (det.detach() > 0)
        return torch.stack([u, v, c / det, -b / det, a / det, torch.sigmoid(p["opacity_logits"]), *rgb])

    def _lists(self):
        """Pairs (tile, Gaussian) sorted by tile and depth: self.gid, and per tile its first pair and length."""
        T, TX, TY = self.T, self.TX, self.TY
        u, v, ca, cb, cc = self.rec[:5].detach()
        lo = lambda x, r, top: ((x - r) / T).floor().clamp(0, top).long()
        hi = lambda x, r, top: (((x + r) / T).floor() + 1).clamp(0, top).long()
        ok = self.seen & torch.isfinite(u) & torch.isfinite(v)
        u0, v0 = torch.where(ok, u, -1e9), torch.where(ok, v, -1e9)
        x0, x1, y0, y1 = lo(u0, self.ext[0], TX), hi(u0, self.ext[0], TX), lo(v0, self.ext[1], TY), hi(v0, self.ext[1], TY)
        wide = (x1 - x0).clamp(min=0)
        cnt = torch.where(ok, wide * (y1 - y0).clamp(min=0), 0)
        g = torch.repeat_interleave(torch.arange(len(cnt), device=DEV), cnt)
        k = torch.arange(len(g), device=DEV) - torch.repeat_interleave(cnt.cumsum(0) - cnt, cnt)
        tx, ty = x0[g] + k % wide[g], y0[g] + k // wide[g]
        U, V, a, b, c = u[g], v[g], ca[g], cb[g], cc[g]
        xl, xh, yl, yh = tx * T + 0.5, tx * T + T - 0.5, ty * T + 0.5, ty * T + T - 0.5
        cl = lambda x, l, h: torch.minimum(torch.maximum(x, l), h)
        Q = lambda X, Y: a * (X - U) ** 2 + 2 * b * (X - U) * (Y - V) + c * (Y - V) ** 2
        best = Q(cl(U, xl, xh), cl(V, yl, yh))
        for X in (xl, xh):
            best = torch.minimum(best, Q(X, cl(V - b / c * (X - U), yl, yh)))
        for Y in (yl, yh):
            best = torch.minimum(best, Q(cl(U - b / a * (Y - V), xl, xh), Y))
        hit = best <= 9.0
        g, tile = g[hit], (ty * TX + tx)[hit]
        rank = torch.empty_like(cnt)
        rank[torch.argsort(self.z.float(), stable=True)] = torch.arange(len(cnt), device=DEV)
        order = torch.argsort(tile * len(cnt) + rank[g])
        self.gid, tile = g[order], tile[order]
        self.len = torch.bincount(tile, minlength=TX * TY)
        self.first = self.len.cumsum(0) - self.len

    def _chunks(self):
        """Groups of tiles of similar length: (tiles, padded list length)."""
        order = torch.argsort(self.len, descending=True)
        lens, at = self.len[order].tolist(), 0
        while at < len(lens) and lens[at] > 0:
            L = lens[at]
            m = max(1, self.CHUNK // (L * self.T * self.T))
            take = [t for t in range(at, min(at + m, len(lens))) if lens[t] > 0]
            yield order[at:at + len(take)], L
            at += len(take)

    def _composite(self, tiles, L, rec):
        """Colours [tiles][T*T][3] of gathered records rec [9][tiles][L]."""
        T, cam = self.T, self.cam
        i = torch.arange(T * T, device=DEV)
        X = ((tiles % self.TX) * T)[:, None] + i % T + 0.5
        Y = ((tiles // self.TX) * T)[:, None] + i // T + 0.5
        u, v, a, b, c, o, r, g, bl = (x[:, None, :] for x in rec)
        dx, dy = X[:, :, None] - u, Y[:, :, None] - v
        live = (torch.arange(L, device=DEV) < self.len[tiles][:, None])[:, None, :]
        alpha = (o * torch.exp(-0.5 * (a * dx * dx + c * dy * dy) - b * dx * dy)).clamp(max=0.99)
        alpha = torch.where(live & (alpha >= 1.0 / 255.0), alpha, 0.0)
        logt = torch.log1p(-alpha)
        after = logt.cumsum(-1)
        alpha = torch.where(after.detach() >= math.log(1e-4), alpha, 0.0)
        logt = torch.where(after.detach() >= math.log(1e-4), logt, 0.0)
        cum = logt.cumsum(-1)
        w = alpha * torch.exp(cum - logt)
        left = torch.exp(cum[..., -1])
        bg = getattr(cam, "bg", (0.0, 0.0, 0.0))
        return torch.stack([(w * x).sum(-1) + left * float(k) for x, k in zip((r, g, bl), bg)], -1)

    def _gather(self, tiles, L):
        at = self.first[tiles][:, None] + torch.arange(L, device=DEV)
        return self.gid[at.clamp(max=len(self.gid) - 1)]

    def image(self):
        T, H, W = self.T, self.cam.height, self.cam.width
        bg = torch.tensor(getattr(self.cam, "bg", (0.0, 0.0, 0.0)), dtype=torch.float64, device=DEV)
        out = bg.expand(self.TX * self.TY, T * T, 3).clone()
        with torch.no_grad():
            for tiles, L in self._chunks():
                out[tiles] = self._composite(tiles, L, self.rec[:, self._gather(tiles, L)])
        out = out.view(self.TY, self.TX, T, T, 3).permute(4, 0, 2, 1, 3).reshape(3, self.TY * T, self.TX * T)
        return out[:, :H, :W].contiguous()

    def backward(self, dL):
        """Gradients of the parameter groups for the upstream gradient dL [3][H][W]."""
        T, H, W = self.T, self.cam.height, self.cam.width
        full = torch.zeros((3, self.TY * T, self.TX * T), dtype=torch.float64, device=DEV)
        full[:, :H, :W] = dL
        up = full.view(3, self.TY, T, self.TX, T).permute(1, 3, 2, 4, 0).reshape(self.TX * self.TY, T * T, 3)
        grad = torch.zeros_like(self.rec)
        for tiles, L in self._chunks():
            gid = self._gather(tiles, L)
            rec = self.rec.detach()[:, gid].requires_grad_()
            (d,) = torch.autograd.grad(self._composite(tiles, L, rec), rec, up[tiles])
            grad.index_add_(1, gid.reshape(-1), d.reshape(9, -1))
        grad = torch.where(self.seen, grad, 0.0)
        got = torch.autograd.grad(self.rec, list(self.leaves.values()), grad)
        return {k: torch.nan_to_num(t) for k, t in zip(self.leaves, got)}


def _l1(image, target):
    d = image - target
    return d.abs().mean(), d.sign() / d.numel(), d.square().sum()


def _dssim(image, target, lam):
    """(1 - lam) L1 + lam (1 - mean SSIM) with an 11-tap Gaussian window: loss, gradient, mean SSIM."""
    x = image.detach().requires_grad_()
    r = torch.arange(-5, 6, dtype=torch.float64, device=DEV)
    w = torch.exp(-r * r / 4.5)
    w = w / w.sum()

    def blur(t):
        H, W = t.shape[-2:]
        p = torch.nn.functional.pad(t, (5, 5))
        t = sum(w[k] * p[..., k:k + W] for k in range(11))
        p = torch.nn.functional.pad(t, (0, 0, 5, 5))
        return sum(w[k] * p[..., k:k + H, :] for k in range(11))

    mx, my = blur(x), blur(target)
    sxx, syy, sxy = blur(x * x) - mx * mx, blur(target * target) - my * my, blur(x * target) - mx * my
    c1, c2 = 0.01 ** 2, 0.03 ** 2
    ssim = ((2 * mx * my + c1) * (2 * sxy + c2) / ((mx * mx + my * my + c1) * (sxx + syy + c2))).mean()
    loss = (1 - lam) * (x - target).abs().mean() + lam * (1 - ssim)
    (g,) = torch.autograd.grad(loss, x)
    return loss.detach(), g, ssim.detach()


def _rows64(groups):
    return torch.cat([groups[k].detach().double().reshape(-1, groups[k].shape[-1])
                      for k in ("means", "log_scales", "quats", "opacity_logits", "sh")])


def _adam64(p, g, m, v, deg, t):
    K = (deg + 1) ** 2
    lr = DECAY * torch.tensor([LR["means"]] * 3 + [LR["log_scales"]] * 3 + [LR["quats"]] * 4 + [LR["opacity_logits"]]
                              + ([LR["dc"]] + [LR["rest"]] * (K - 1)) * 3, dtype=torch.float64, device=DEV)[:, None]
    m = B1 * m.double() + (1 - B1) * g
    v = B2 * v.double() + (1 - B2) * g * g
    p = p - lr * (m / (1 - B1 ** t)) / ((v / (1 - B2 ** t)).sqrt() + EPS)
    return p, m, v


def _exact_views(groups, cams, targets, tile):
    """Sum over views of the gradient [rows][n] of each view's mean L1."""
    total = 0
    for cam, target in zip(cams, targets):
        r = _Raster64(groups, cam, tile)
        total = total + _rows64(r.backward(_l1(r.image(), target.double())[1]))
    return total


def _exact_init(case, seed):
    """The network's features and the seeding from the exact neighbours."""
    pts = prepare(case, seed)["points"]
    n, P = pts.shape[1], pts.t().contiguous()
    P64 = P.double()
    nb = torch.empty((n, 32), dtype=torch.long, device=DEV)
    for at in range(0, n, 4096):
        near = torch.cdist(P[at:at + 4096], P).topk(49, largest=False).indices
        d = (P64[near] - P64[at:at + 4096, None]).square().sum(-1)
        d[near == torch.arange(at, min(at + 4096, n), device=DEV)[:, None]] = math.inf
        nb[at:at + 4096] = near.gather(1, d.argsort(1)[:, :32])

    def eig(k):
        q = P64[nb[:, :k]]
        q = q - q.mean(1, keepdim=True)
        cov = (q.transpose(1, 2) @ q / k).cpu()
        w, V = (t.to(DEV) for t in torch.linalg.eigh(cov))
        big = V.abs().argmax(1, keepdim=True)
        return w, V * V.gather(1, big).sign()

    w, V = eig(32)
    off = P64[nb] - P64[:, None]
    md = off.norm(dim=-1).mean(1)
    features = torch.cat([w / w.sum(1, keepdim=True), V.transpose(1, 2).reshape(n, 9), off.mean(1) / md[:, None],
                          -3 * md.log()[:, None]], 1)
    nrm = eig(16)[1][:, :, 0]
    st = off[:, :3].norm(dim=-1).mean(1)
    qw = (0.5 * (1 + nrm[:, 2])).sqrt()
    z = torch.zeros_like(qw)
    K = (case["deg"] + 1) ** 2
    rows = [*P64.t(), st.log(), st.log(), (float(np.float32(0.1)) * st).log(), qw, -nrm[:, 1] / (2 * qw),
            nrm[:, 0] / (2 * qw), z, z + math.log(0.1 / 0.9)]
    return {"params": torch.cat([torch.stack(rows), torch.zeros((3 * K, n), dtype=torch.float64, device=DEV)]),
            "features": features, "features_bf16": features, "frame_q": None, "nb": None}


def _net64(seed):
    """The network's starting parameters: Glorot-uniform matrices, zero biases."""
    g = torch.Generator(device="cpu").manual_seed(seed)
    out = []
    for o, i in ((64, 16), (64, 64), (8, 64)):
        W = (torch.rand((o, i), generator=g) * 2 - 1) * math.sqrt(6.0 / (i + o))
        out += [W.to(DEV), torch.zeros(o, device=DEV)]
    return out


def _forward64(net, x):
    gelu = lambda z: 0.5 * z * (1 + torch.erf(z / math.sqrt(2.0)))
    W = [t.to(torch.bfloat16).double() if t.dim() == 2 and not t.requires_grad else t for t in net]
    h = gelu(x @ W[0].t() + W[1])
    h = gelu(h @ W[2].t() + W[3])
    return h @ W[4].t() + W[5]


def _exact_fit(case, seed):
    x, t = _mlp_rows(case["n"], seed)
    net = _net64(seed)
    low = [w.to(torch.bfloat16).double().requires_grad_() if w.dim() == 2 else w.double().requires_grad_() for w in net]
    y, t = _forward64(low, x.double()), t.double()
    q = y[:, 3:7] / y[:, 3:7].norm(dim=1, keepdim=True)
    f = (q * t[:, 3:7]).sum(1)
    loss = ((y[:, :3] - t[:, :3]).square().sum(1) + 1 - f * f + (y[:, 7] - t[:, 7]).square()).sum()
    g = torch.cat([d.reshape(-1) for d in torch.autograd.grad(loss / case["n"], low)])
    m, v = 0.1 * g, 0.001 * g * g
    # a first Adam step moves every weight by the learning rate in its gradient's sign: the moments say more
    return {"loss": loss.detach(), "master": None, "m": m, "v": v}


def _exact_ba(case, seed):
    R, t, P, cam, pt, uv, K = _ba_problem(case, seed)
    R, t, P, uv, cam, pt = R.double(), t.double(), P.double(), uv.double(), cam.long(), pt.long()
    C, n, sigma, delta = case["cams"], case["points"], 0.5, 2.0
    skew = lambda a: torch.stack([torch.zeros_like(a[:, 0]), -a[:, 2], a[:, 1], a[:, 2], torch.zeros_like(a[:, 0]),
                                  -a[:, 0], -a[:, 1], a[:, 0], torch.zeros_like(a[:, 0])], 1).view(-1, 3, 3)

    def terms(R, t, P):
        rp = torch.einsum("mij,mj->mi", R[cam], P[pt])
        x = rp + t[cam]
        r = torch.stack([K[0] * x[:, 0] / x[:, 2] + K[2], K[1] * x[:, 1] / x[:, 2] + K[3]], 1) - uv
        e = r.norm(dim=1) / sigma
        seen = x[:, 2] > 1e-6
        rho = torch.where(e <= delta, e * e, 2 * delta * e - delta * delta)
        w = torch.where(e <= delta, 1.0, delta / e.clamp(min=1e-300))
        return rp, x, r, torch.where(seen, w, 0.0), torch.where(seen, rho, 0.0).sum()

    base = R[1] @ (-(R[1].t() @ t[1]) + R[0].t() @ t[0])
    fixed = torch.zeros((C, 6), dtype=torch.bool, device=DEV)
    fixed[0] = True
    fixed[1, 3 + int(base.abs().argmax())] = True
    fixed = fixed.reshape(-1)
    # pairs of observations of one point, for the camera blocks it couples
    cnt = torch.bincount(pt, minlength=n)
    first = cnt.cumsum(0) - cnt
    a = torch.repeat_interleave(torch.arange(len(pt), device=DEV), cnt[pt])
    b = first[pt[a]] + torch.arange(len(a), device=DEV) - torch.repeat_interleave(cnt[pt].cumsum(0) - cnt[pt], cnt[pt])
    lam, state = 1e-4, terms(R, t, P)
    costs = [state[4]]
    for _ in range(case["iters"]):
        rp, x, r, w, cost = state
        iz = 1 / x[:, 2]
        D = torch.zeros((len(pt), 2, 3), dtype=torch.float64, device=DEV)
        D[:, 0, 0], D[:, 0, 2] = K[0] * iz, -K[0] * x[:, 0] * iz * iz
        D[:, 1, 1], D[:, 1, 2] = K[1] * iz, -K[1] * x[:, 1] * iz * iz
        Jc = torch.cat([D @ -skew(rp), D], 2)
        Jp = D @ R[cam]
        W = (w / sigma ** 2)[:, None, None]
        add = lambda size, at, v: torch.zeros((size, *v.shape[1:]), dtype=torch.float64, device=DEV).index_add_(0, at, v)
        Hc, Hp = add(C, cam, W * Jc.transpose(1, 2) @ Jc), add(n, pt, W * Jp.transpose(1, 2) @ Jp)
        bc, bp = add(C, cam, -(W * Jc.transpose(1, 2) @ r[..., None])), add(n, pt, -(W * Jp.transpose(1, 2) @ r[..., None]))
        Hcp = W * Jc.transpose(1, 2) @ Jp
        damp = lambda H: H + lam * torch.diag_embed(torch.diagonal(H, dim1=1, dim2=2))
        Hi = torch.linalg.inv(torch.where((cnt > 0)[:, None, None], damp(Hp), torch.eye(3, dtype=torch.float64, device=DEV)))
        E = Hcp @ Hi[pt]
        Sm = add(C * C, cam[a] * C + cam[b], -(E[a] @ Hcp[b].transpose(1, 2)))
        Sm[torch.arange(C, device=DEV) * (C + 1)] += damp(Hc)
        Sm = Sm.view(C, C, 6, 6).permute(0, 2, 1, 3).reshape(6 * C, 6 * C)
        rhs = (bc - add(C, cam, E @ bp[pt])).reshape(-1)
        free = ~fixed & (torch.diagonal(Sm) > 0)
        dc = torch.zeros(6 * C, dtype=torch.float64, device=DEV)
        dc[free] = torch.linalg.solve(Sm[free][:, free], rhs[free])
        dc = dc.view(C, 6)
        dp = (Hi @ (bp - add(n, pt, Hcp.transpose(1, 2) @ dc[cam][..., None])))[..., 0]
        new = terms(torch.linalg.matrix_exp(skew(dc[:, :3])) @ R, t + dc[:, 3:], P + dp)
        if bool(new[4] < cost):
            R, t, P, state, lam = torch.linalg.matrix_exp(skew(dc[:, :3])) @ R, t + dc[:, 3:], P + dp, new, lam / 10
        else:
            lam *= 10
        costs.append(state[4])
    return {"R": R, "t": t, "P": P, "costs": torch.stack(costs)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        groups, cam, target = _scene(case, seed)
        r = _Raster64(groups, cam, case["tile"])
        image, target = r.image(), target.double()
        if case["dssim"]:
            loss, dL, ssim = _dssim(image, target, case["dssim"])
            losses = torch.stack([loss, ssim])
        else:
            l1, dL, sse = _l1(image, target)
            losses = torch.stack([l1, sse])
        g = _rows64(r.backward(dL))
        p, m, v = _adam64(_rows64(groups), g, *_moments(case["n"], case["deg"], seed), case["deg"], ADAM_T + 1)
        return {"loss": losses, "image": image, "params": p, "m": m, "v": v}
    if kind == "render":
        groups, cam, _ = _scene(case, seed)
        return {"image": _Raster64(groups, cam, case["tile"]).image()}
    if kind == "autograd":
        groups, cam, target = _scene(case, seed)
        r = _Raster64(groups, cam, case["tile"])
        image = r.image()
        d = image - target.double()
        return {"loss": d.square().mean(), "image": image, "grads": r.backward(2 * d / d.numel())}
    if kind == "batch":
        out = {"params": [], "m": [], "v": []}
        for k, (groups, cams, targets) in enumerate(_batch_scenes(case, seed)):
            g = _exact_views(groups, cams, targets, case["tile"])
            mom = _moments(groups["means"].shape[1], case["deg"], seed + k)
            for name, t in zip(("params", "m", "v"), _adam64(_rows64(groups), g, *mom, case["deg"], 1)):
                out[name].append(t)
        return out
    if kind == "init":
        return _exact_init(case, seed)
    if kind == "mlp":
        x, _ = _mlp_rows(case["n"], seed)
        net = [t.double() if t.dim() == 1 else t for t in _net64(seed)]
        return {"y": torch.cat([_forward64(net, c.double()) for c in x.split(1 << 19)])}
    if kind == "fit":
        return _exact_fit(case, seed)
    if kind == "ba":
        return _exact_ba(case, seed)
    return None  # the stereo depth follows from integer costs that float32 decisions fix: no 64-bit value
