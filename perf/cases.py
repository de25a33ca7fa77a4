"""The work a user of this framework has it do, as cases that can be timed: tracking a camera
against a map, rendering it, differentiating it, optimising it over a window of keyframes,
adding and removing Gaussians, and measuring a render's quality -- each through the public
entry points of paper_2408_05635_gb300.

    prepare(case, seed)  the inputs on the GPU and what a program keeps between calls
                         (contexts, workspaces, planned problems)
    run(state)           one pass through the public calls, and its outputs
    exact(case, seed)    the same outputs in plain torch in 64 bits, where that is quick

Scenes are the synthetic ones of the tests and the benchmark (a cube of Gaussians in front
of the camera; a textured room), drawn on the GPU, and the map a keyframe builds (a Gaussian
per pixel of an RGB-D frame).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2408_05635_gb300 import autograd, gs, scenes, slam

DEV = "cuda"
DTYPES = {"fp32": torch.float32, "bf16": torch.bfloat16, "fp16": torch.float16}
ATTRIBUTES = ("means", "quats", "log_scales", "logits", "rgb")
IMAGES = [(320, 240), (640, 480), (1200, 680)]  # the keyframe sizes of the batched workload


def _case(name, kind, **over):
    """scene: cube | room | frames (a Gaussian per pixel of the first keyframe, and of a
    quarter of the pixels of the others); n: Gaussians (of cube and room); frames: views or
    keyframes (mixed: their sizes alternate over IMAGES); hyps: pose hypotheses per frame;
    iters: tracking iterations per call; fused: the launch schedule's fused compositor."""
    c = {"kind": kind, "scene": "room", "n": 200_000, "width": 640, "height": 480, "frames": 1, "mixed": False,
         "hyps": 1, "iters": 1, "dtype": "fp32", "isotropic": False, "fused": False}
    c.update(over)
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest call: one tracking iteration of a thumbnail against a toy map (what a
        # test, a demo or a coarse relocalisation level calls); launches and latency
        _case("track_160x120_2k", "track", scene="cube", n=2_000, width=160, height=120),
        # a camera frame in pinned host memory, one iteration per call, pose and loss read
        # back: tracking end to end at the 640 x 480 / 200k size
        _case("upload_640x480_200k", "upload", fused=True),
        # the sequence driver's tracking of a frame (several iterations in one graph, status
        # read back), default launch schedule
        _case("frame_640x480_200k", "frame", iters=4),
        # the long sequence's map: 2M Gaussians in FP16
        _case("track_640x480_2M_fp16", "track", n=2_000_000, iters=2, dtype="fp16", fused=True),
        # pose hypotheses on keyframes of uneven resolution in one call, BF16 attributes
        _case("hypotheses_12_bf16", "track", n=500_000, frames=6, mixed=True, hyps=2, iters=2, dtype="bf16", fused=True),
        # novel-view synthesis: forward only, a large map and image
        _case("render_1200x680_1M", "render", n=1_000_000, width=1200, height=680),
        # the isotropic Gaussian of Eq. 1 as printed, low-precision attributes, an odd image
        _case("render_333x257_iso_bf16", "render", n=30_000, width=333, height=257, dtype="bf16", isotropic=True),
        # an optimisation written in torch around the differentiable renderer: odd image,
        # forward and backward to every parameter and the pose
        _case("autograd_317x241_60k", "autograd", n=60_000, width=317, height=241),
        # the mapping step's gradients over a window of eight wide keyframes (the largest)
        _case("window_8x1200x680_1M", "window", n=1_000_000, width=1200, height=680, frames=8),
        # the same on the kind of map the sequence driver builds: a Gaussian per pixel
        _case("window_4x640x480_dense", "window", scene="frames", frames=4),
        # the map side of a keyframe: add its new pixels, one Adam step, remove the faded
        _case("map_640x480_1M_fp16", "map", n=1_000_000, dtype="fp16"),
        # evaluating a rendered keyframe: PSNR and depth sums, MS-SSIM
        _case("quality_640x480", "quality"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["track", "track", "upload", "frame", "render", "autograd", "window", "window", "map", "quality"])
    width = _log(rng, 96, 1200)
    height = max(64, int(width * rng.uniform(0.55, 0.78)))
    c = _case(None, kind, n=_log(rng, 1_500, 1_200_000), width=width, height=height)
    if kind in ("track", "upload", "frame"):
        c["fused"] = rng.random() < 0.6
        c["dtype"] = rng.choice(["fp32", "fp32", "bf16", "fp16"])
        c["isotropic"] = rng.random() < 0.2
    if kind == "frame":
        c["iters"] = rng.randint(2, 4)
    if kind == "track":
        c["frames"], c["hyps"] = rng.choice([(1, 1), (1, 1), (1, 5), (3, 2), (5, 3)])
        c["mixed"] = c["frames"] > 1
        c["iters"] = 2 if c["frames"] * c["hyps"] > 1 else rng.randint(1, 2)
    if kind in ("render", "autograd"):
        c["dtype"] = rng.choice(["fp32", "fp32", "bf16"]) if kind == "render" else "fp32"
        c["isotropic"] = kind == "render" and rng.random() < 0.3
        c["frames"] = rng.choice([1, 1, 2])
    if kind == "window":
        c["frames"] = rng.randint(2, 8)
        c["scene"] = rng.choice(["room", "frames"])
        if c["scene"] == "frames":
            c["width"] = min(c["width"], 800)
            c["height"] = min(c["height"], 600)
            c["frames"] = min(c["frames"], 4)
    if kind == "map":
        c["dtype"] = rng.choice(["fp32", "bf16", "fp16"])
        c["isotropic"] = rng.random() < 0.3
    if kind == "quality":  # the coarsest of five scales holds one 11 x 11 window
        c["width"] = max(176, c["width"])
        c["height"] = max(176, c["height"])
    if kind in ("track", "render") and c["frames"] == 1 and c["n"] < 4_000:
        c["scene"] = "cube"
    return c


# --------------------------------------------------------------------------- inputs


def _camera(width, height, scene="room"):
    f = {"cube": 0.875}.get(scene, 525.0 / 640.0) * width
    return scenes.Cam(f, f, (width - 1) / 2.0, (height - 1) / 2.0, width, height)


def _room(n, seed):
    """scenes.room_scene's distribution drawn on the GPU, along a Morton curve of the means."""
    gen = torch.Generator(DEV).manual_seed(seed)
    rects = scenes.room_rects(seed)
    area = torch.tensor([r.su * r.sv for r in rects], device=DEV)
    which = torch.multinomial(area, n, replacement=True, generator=gen)
    table = lambda f: torch.tensor(np.stack([np.atleast_1d(f(r)) for r in rects]), dtype=torch.float32, device=DEV)[which]
    a = torch.rand(n, 1, device=DEV, generator=gen) * table(lambda r: r.su)
    b = torch.rand(n, 1, device=DEV, generator=gen) * table(lambda r: r.sv)
    jitter = 0.005 * torch.randn(n, 1, device=DEV, generator=gen)
    means = table(lambda r: r.origin) + a * table(lambda r: r.u) + b * table(lambda r: r.v) + jitter * table(lambda r: r.normal)
    phase = table(lambda r: r.phase)
    wave = 0.15 * torch.sin(2 * math.pi * a / 1.7 + phase) * torch.sin(2 * math.pi * b / 1.3 + 0.5 * phase)
    checker = ((torch.floor(a / 0.5) + torch.floor(b / 0.5)) % 2) * 0.12 - 0.06
    rgb = (table(lambda r: r.base) + wave + checker).clamp(0.0, 1.0)
    cell = torch.floor((means - means.amin(0)) / 0.01).to(torch.int64)
    code = torch.zeros(n, dtype=torch.int64, device=DEV)
    for bit in range(10):
        for axis in range(3):
            code |= ((cell[:, axis] >> bit) & 1) << (3 * bit + axis)
    order = torch.argsort(code, stable=True)
    return {"means": means[order], "quats": torch.randn(n, 4, device=DEV, generator=gen),
            "log_scales": -4.0 + 0.4 * torch.randn(n, 3, device=DEV, generator=gen),
            "logits": 2.0 + torch.randn(n, device=DEV, generator=gen), "rgb": rgb[order]}


def _cube(n, seed):
    """scenes.cube_scene's distribution."""
    g, _ = scenes.cube_scene(n, seed)
    return {k: torch.as_tensor(v, device=DEV) for k, v in zip(ATTRIBUTES, g.arrays())}


def _dense_count(px, frames):
    """Gaussians of the map keyframes build (some pixels look out of the open ceiling)."""
    return int(0.7 * px * (1 + 0.25 * (frames - 1)))


def _from_frames(frames, cam, seed):
    """The map keyframes build: a Gaussian one pixel wide per pixel with depth of the first,
    and of a quarter of the pixels of the others, in pixel order; _dense_count of them."""
    gen = torch.Generator(DEV).manual_seed(seed)
    means, rgbs, scales = [], [], []
    v, u = torch.meshgrid(torch.arange(cam.height, device=DEV), torch.arange(cam.width, device=DEV), indexing="ij")
    for k, (pose, rgb, depth) in enumerate(frames):
        keep = depth > 0
        if k:
            keep &= torch.rand(depth.shape, device=DEV, generator=gen) < 0.25
        d = depth[keep].double()
        local = torch.stack([(u[keep] - cam.cx) / cam.fx * d, (v[keep] - cam.cy) / cam.fy * d, d], 1)
        R, t = scenes.pose_rt(pose)
        means.append(((local - torch.tensor(t, device=DEV)) @ torch.tensor(R, device=DEV)).float())
        rgbs.append(rgb[:, keep].T)
        scales.append(torch.log(d / cam.fx).float())
    means, rgb, ls = torch.cat(means), torch.cat(rgbs), torch.cat(scales)
    n = _dense_count(cam.width * cam.height, len(frames))
    pick = torch.randperm(means.shape[0], device=DEV, generator=gen)
    pick = pick[torch.arange(n, device=DEV) % pick.numel()].sort().values
    means, rgb, ls = means[pick], rgb[pick], ls[pick]
    quats = torch.tensor([1.0, 0.0, 0.0, 0.0], device=DEV) + 0.05 * torch.randn(n, 4, device=DEV, generator=gen)
    return {"means": means, "quats": quats, "logits": 1.0 + torch.randn(n, device=DEV, generator=gen),
            "log_scales": ls[:, None] + 0.1 * torch.randn(n, 3, device=DEV, generator=gen),
            "rgb": (rgb + 0.02 * torch.randn(n, 3, device=DEV, generator=gen)).clamp(0.0, 1.0)}


def _observe(pose, cam, scene, gen, seed):
    """An RGB-D frame with its depth prior: the ray-cast room (the cube scene gets a smooth
    colour pattern and a slanted depth)."""
    if scene == "cube":
        v, u = torch.meshgrid(torch.arange(cam.height, device=DEV), torch.arange(cam.width, device=DEV), indexing="ij")
        rgb = torch.stack([0.5 + 0.4 * torch.sin(0.05 * u + k + 0.04 * v) for k in range(3)])
        depth = 1.5 + 0.002 * u.float() + 0.003 * v.float()
    else:
        rgb, depth = scenes.raycast_room_torch(pose, cam, seed, DEV)
    noise = 1.0 + 0.02 * torch.randn(depth.shape, device=DEV, generator=gen)
    hole = torch.rand(depth.shape, device=DEV, generator=gen) < 0.05
    return rgb, depth, torch.where(hole, torch.zeros_like(depth), depth * noise)


def _inputs(case, seed):
    """Gaussians, per view its camera, pose and RGB-D targets: everything a pass reads."""
    rng, gen = np.random.default_rng(seed), torch.Generator(DEV).manual_seed(seed + 1)
    scene, kind, V = case["scene"], case["kind"], case["frames"]
    sizes = [IMAGES[k % 3] if case["mixed"] else (case["width"], case["height"]) for k in range(V)]
    cams = [_camera(w, h, scene) for w, h in sizes]
    if scene == "cube":
        truth = [scenes.identity_pose()] * V
    elif scene == "frames":
        truth = scenes.spline_trajectory(200, seed)[:4 * V:4]
    elif kind == "window":
        truth = scenes.mapping_keyframes(max(V, 2))[:V]
    elif V == 1:
        truth = [scenes.perturb_pose(scenes.tracking_gt_pose(), rng, 5.0, 0.1)]
    else:
        truth = scenes.batched_keyframes(V, 1, seed)[3]
    views = [_observe(p, c, scene, gen, seed) for p, c in zip(truth, cams)]
    if scene == "cube":
        g = _cube(case["n"], seed)
    elif scene == "frames":
        g = _from_frames([(p, rgb, d) for p, (rgb, d, _) in zip(truth, views)], cams[0], seed)
    else:
        g = _room(case["n"], seed)
    if case["isotropic"]:
        g["quats"], g["log_scales"] = None, g["log_scales"].mean(1)
    dt = DTYPES[case["dtype"]] if kind != "map" else torch.float32
    g = {k: v if v is None or k == "means" else v.to(dt).contiguous() for k, v in g.items()}
    poses, flat_cams, flat_views = [], [], []
    for p, c, v in zip(truth, cams, views):
        for _ in range(case["hyps"]):
            poses.append(scenes.jitter_pose(p, rng, 2.0, 0.04) if case["hyps"] > 1 else
                         scenes.perturb_pose(p, rng, 2.0, 0.05) if kind in ("track", "upload", "frame") else
                         scenes.perturb_pose(p, rng, 0.3, 0.01))
            flat_cams.append(c)
            flat_views.append(v)
    poses = torch.tensor(np.stack(poses), dtype=torch.float64, device=DEV)
    return g, flat_cams, poses, flat_views


def _upstream(cams, seed):
    """dL/d(rgb, depth, silhouette) of some loss on the maps."""
    gen = torch.Generator(DEV).manual_seed(seed + 2)
    P = sum(c.width * c.height for c in cams)
    return tuple(torch.randn(k * P, device=DEV, generator=gen) for k in (3, 1, 1))


def _concat(views, k):
    return torch.cat([v[k].reshape(-1) for v in views])


# --------------------------------------------------------------------------- one pass


def prepare(case, seed):
    kind = case["kind"]
    g, cams, poses, views = _inputs(case, seed)
    s = {"case": case, "cams": cams, "poses": poses, "views": views}
    if kind == "quality":
        return _prepare_quality(s, seed)
    if kind == "map":
        return _prepare_map(s, g, seed)
    s["g"] = gs.GaussianTensors(*(g[k] for k in ATTRIBUTES))
    if kind == "frame":
        s["tracker"] = slam.Tracker(cams[0], case["iters"])
        if case["fused"]:
            s["tracker"].R.set_schedule(flags=gs.GS_SCHED_FUSED)
        return s
    s["R"] = gs.Rasterizer()
    if case["fused"]:
        s["R"].set_schedule(flags=gs.GS_SCHED_FUSED)
    if kind == "autograd":
        s["up"] = _upstream(cams, seed)
        return s
    s["prob"] = s["R"].plan(s["g"], cams, poses, margin=1.5)
    if kind == "render":
        return s
    if kind == "window":
        s["targets"] = [tuple(x.reshape(-1).contiguous() for x in v) for v in views]
        return s
    s["ws"], s["nb"] = s["R"].workspace(s["prob"])
    V = len(cams)
    s["pose"], s["adam"] = poses.clone(), torch.zeros(V, 16, dtype=torch.float64, device=DEV)
    s["hist"] = torch.zeros(case["iters"], V, dtype=torch.float64, device=DEV)
    s["targets"] = [_concat(views, k) for k in range(3)]
    if kind == "upload":  # the camera's frame lands in pinned host memory
        s["host"] = [t.cpu().pin_memory() for t in s["targets"]]
        s["result"] = torch.zeros(V, 8, dtype=torch.float64).pin_memory()
        s["src"] = gs.gs_host_targets(*(t.data_ptr() for t in s["host"]), s["result"].data_ptr())
    return s


def _prepare_quality(s, seed):
    gen = torch.Generator(DEV).manual_seed(seed + 3)
    rgb, depth, _ = s["views"][0]
    blur = torch.nn.functional.avg_pool2d(rgb[None], 3, 1, 1)[0]
    s["obs"] = (rgb.reshape(-1).contiguous(), depth.reshape(-1).contiguous())
    s["img"] = ((blur + 0.01 * torch.randn(rgb.shape, device=DEV, generator=gen)).reshape(-1).contiguous(),
                (depth * (1 + 0.005 * torch.randn(depth.shape, device=DEV, generator=gen))).reshape(-1).contiguous())
    s["sums"], s["ssim"] = (torch.zeros(4, dtype=torch.float64, device=DEV) for _ in range(2))
    return s


def _map_inputs(s, g, seed):
    """The live map with some Gaussians faded, gradients of a mapping step, a silhouette."""
    gen = torch.Generator(DEV).manual_seed(seed + 3)
    n, cam = g["means"].shape[0], s["cams"][0]
    g = dict(g)
    faded = torch.rand(n, device=DEV, generator=gen) < 0.08
    g["logits"] = torch.where(faded, -7.0 + 0.1 * torch.randn(n, device=DEV, generator=gen), g["logits"])
    sil = torch.nn.functional.interpolate(torch.rand(1, 1, 9, 12, device=DEV, generator=gen), (cam.height, cam.width),
                                          mode="bilinear")[0, 0].contiguous()
    cap = (n + cam.width * cam.height + 3) // 4 * 4
    grads = {k: torch.randn((cap,) + v.shape[1:], device=DEV, generator=gen) * 0.1 for k, v in g.items() if v is not None}
    return g, sil, cap, grads


def _prepare_map(s, g, seed):
    case = s["case"]
    g, sil, cap, s["grads"] = _map_inputs(s, g, seed)
    lowp = DTYPES[case["dtype"]] if case["dtype"] != "fp32" else None
    s["n"], s["sil"] = g["means"].shape[0], sil
    s["map"], s["spare"] = (gs.Map(cap, DEV, lowp_dtype=lowp, isotropic=case["isotropic"]) for _ in range(2))
    s["map"].load(gs.GaussianTensors(*(g[k] for k in ATTRIBUTES)))
    return s


def run(s):
    return {"track": _run_track, "upload": _run_track, "frame": _run_frame, "render": _run_render,
            "autograd": _run_autograd, "window": _run_window, "map": _run_map, "quality": _run_quality}[s["case"]["kind"]](s)


def _run_track(s):
    R, iters = s["R"], s["case"]["iters"]
    s["pose"].copy_(s["poses"])
    s["adam"].zero_()
    if "src" in s:
        gs.gs_track_step_upload(R.ctx, s["prob"], s["g"].c(), None, s["src"], s["pose"], s["adam"], s["hist"], iters,
                                s["ws"], s["nb"])
    else:
        tg = gs.gs_targets(*(t.data_ptr() for t in s["targets"]))
        gs.gs_track_step(R.ctx, s["prob"], s["g"].c(), tg, s["pose"], s["adam"], s["hist"], iters, s["ws"], s["nb"])
    out = {"pose": s["pose"], "loss": s["hist"]}
    if "src" in s:
        out["result"] = s["result"]
    return out


def _run_frame(s):
    t = s["tracker"]
    return {"pose": t.track(s["g"], s["poses"][0], *s["views"][0]), "loss": t.hist}


def _run_render(s):
    return s["R"].render(s["prob"], s["g"], s["poses"])


def _run_autograd(s):
    g = s["g"]
    leaves = [t.detach().requires_grad_(True) for t in (g.means, g.quats, g.log_scales, g.logits, g.rgb)]
    tangent = torch.zeros(len(s["cams"]), 6, dtype=torch.float64, device=DEV, requires_grad=True)
    maps = autograd.render(s["R"], *leaves, s["cams"], s["poses"], tangent)
    grads = torch.autograd.grad(maps, leaves, s["up"])
    return {"maps": [m.detach() for m in maps], "grads": dict(zip(ATTRIBUTES, grads))}


def _run_window(s):
    V = len(s["cams"])
    return s["R"].mapping_grads(s["g"], s["cams"], s["poses"], s["targets"], chunk=V, probs=[s["prob"]])


def _run_map(s):
    m, spare = s["map"], s["spare"]
    m.count.fill_(s["n"])
    rgb, depth, _ = s["views"][0]
    m.add_from_frame(s["cams"][0], s["poses"][0], rgb, depth, s["sil"])
    m.adam_step(s["grads"], 1)
    m.prune_into(spare)
    return {"map": spare.p, "copy": spare.lp, "moments": spare.state, "count": spare.count}


def _run_quality(s):
    cam = s["cams"][0]
    gs.gs_image_metrics(*s["img"], *s["obs"], s["sums"])
    gs.gs_msssim(s["img"][0], s["obs"][0], cam.width, cam.height, s["ssim"])
    return {"sums": s["sums"], "ssim": s["ssim"]}


# --------------------------------------------------------------------------- what a pass cannot do without

FLOP_PROJECT, FLOP_FORWARD, FLOP_BACKWARD = 150, 23, 58  # per Gaussian and view; per (pixel, Gaussian) pair


def work(case):
    """bytes: every parameter and image read once, every output written once.  flops: the
    projection of every Gaussian in every view and the (pixel, Gaussian) pairs that
    contribute (counted on some of the scenes: 36 per pixel of the room at 200k, 16 at 60k,
    62 at 2M; 14 of the 2k cube; 38 of the dense maps)."""
    kind = case["kind"]
    sizes = [IMAGES[k % 3] if case["mixed"] else (case["width"], case["height"]) for k in range(case["frames"])]
    P = sum(w * h for w, h in sizes) * case["hyps"]
    V = case["frames"] * case["hyps"]
    px = case["width"] * case["height"]
    if kind == "quality":
        # five statistics over an 11 x 11 window (separable: 2 x 11 taps) at 4/3 px positions
        return {"bytes": 32 * px, "flops": 4 / 3 * px * 3 * 2 * 22 * 5}
    n = case["n"] if case["scene"] != "frames" else _dense_count(px, case["frames"])
    w = 8 if case["isotropic"] else 14
    if kind == "map":
        live = n + px // 2
        low = 0 if case["dtype"] == "fp32" else 2 * (w - 3)
        # add: the frame read, half of it written; Adam: parameter, gradient and two moments
        # read, three written; removal: parameters, moments and copies read and written
        return {"bytes": 24 * px + (12 * w + low) * px // 2 + (28 * w + low) * live + 2 * (12 * w + low) * live,
                "flops": 12 * w * live}
    attr = 12 + (w - 3) * (4 if case["dtype"] == "fp32" else 2)
    per_pixel = {"cube": 14.0 * n / 2_000, "frames": 38.0}.get(
        case["scene"], 36.0 * (n / 2e5) ** (0.6 if n < 200_000 else 0.25))
    pairs = per_pixel * P
    if kind == "render":
        return {"bytes": n * attr + 20 * P, "flops": FLOP_PROJECT * n * V + FLOP_FORWARD * pairs}
    if kind in ("autograd", "window"):
        maps = 40 if kind == "autograd" else 20  # maps out and upstream in, or targets in
        return {"bytes": 2 * n * attr + maps * P,
                "flops": 2 * FLOP_PROJECT * n * V + (FLOP_FORWARD + FLOP_BACKWARD) * pairs}
    targets = 20 * P
    return {"bytes": case["iters"] * (n * attr + targets),
            "flops": case["iters"] * (2 * FLOP_PROJECT * n * V + (FLOP_FORWARD + FLOP_BACKWARD) * pairs)}


# --------------------------------------------------------------------------- in 64 bits

ALPHA_MIN, ALPHA_MAX, T_MIN, Z_NEAR, JAC_CLIP, SIL = 1.0 / 255.0, 0.99, 1e-4, 0.2, 1.3, 0.99
W_RGB, W_DEPTH, W_VIS, W_PRIOR = 0.5, 1.0, 0.1, 0.5
TILE = 32


def _rotation(q):
    w, x, y, z = (q / q.norm(dim=-1, keepdim=True)).unbind(-1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], -1).reshape(q.shape[:-1] + (3, 3))


def _screen(g, cam, pose, tangent):
    """Screen quantities of the Gaussians that reach the view, n x 10 (mean 2, depth, opacity,
    conic 3, colour 3), and their support half-extents; differentiable in g and in the pose's
    tangent (rotation about the camera centre, shift)."""
    W, t = _rotation(pose[:4]), pose[4:]
    k = tangent[:3]
    zero = torch.zeros_like(k[0])
    skew = torch.stack([zero, -k[2], k[1], k[2], zero, -k[0], -k[1], k[0], zero]).reshape(3, 3)
    turn = torch.eye(3, dtype=torch.float64, device=DEV) + skew
    xc = (g["means"] @ W.T + t) @ turn.T + tangent[3:]
    at = (xc[:, 2] > Z_NEAR).nonzero()[:, 0]
    x, y, z = xc[at].unbind(1)
    scale = torch.exp(g["log_scales"][at]).reshape(at.numel(), -1).expand(-1, 3)
    M = turn @ W if g["quats"] is None else turn @ W @ _rotation(g["quats"][at])
    M = M * scale[:, None, :]
    lim_x, lim_y = JAC_CLIP * 0.5 * cam.width / cam.fx, JAC_CLIP * 0.5 * cam.height / cam.fy
    tx, ty = (x / z).clamp(-lim_x, lim_x), (y / z).clamp(-lim_y, lim_y)
    n0 = (cam.fx / z)[:, None] * M[:, 0] - (cam.fx * tx / z)[:, None] * M[:, 2]
    n1 = (cam.fy / z)[:, None] * M[:, 1] - (cam.fy * ty / z)[:, None] * M[:, 2]
    a, b, c = (n0 * n0).sum(1), (n0 * n1).sum(1), (n1 * n1).sum(1)
    det = torch.linalg.cross(n0, n1).square().sum(1)
    o = torch.sigmoid(g["logits"][at])
    q = torch.stack([cam.fx * x / z + cam.cx, cam.fy * y / z + cam.cy, z, o, c / det, -b / det, a / det], 1)
    q = torch.cat([q, g["rgb"][at]], 1)
    with torch.no_grad():
        r2 = 2 * torch.log(o / ALPHA_MIN).clamp_min(0)
        half = torch.stack([(r2 * a).sqrt(), (r2 * c).sqrt()], 1) + 1.0
        mean = q[:, :2]
        size = torch.tensor([cam.width - 1.0, cam.height - 1.0], dtype=torch.float64, device=DEV)
        ok = (o >= ALPHA_MIN) & (det > 0) & ((mean + half) >= 0).all(1) & ((mean - half) <= size).all(1)
        keep = ok.nonzero()[:, 0]
        keep = keep[torch.argsort(q[keep, 2], stable=True)]
    return q[keep], half[keep]


def _composite(q, u, v):
    """Eqs. 2-4 at pixels (u, v) over depth-sorted screen Gaussians: maps of 5 rows."""
    dx, dy = u[:, None] - q[:, 0], v[:, None] - q[:, 1]
    alpha = q[:, 3] * torch.exp(-0.5 * (q[:, 4] * dx * dx + 2 * q[:, 5] * dx * dy + q[:, 6] * dy * dy))
    alpha = torch.where(alpha >= ALPHA_MIN, alpha.clamp(max=ALPHA_MAX), torch.zeros_like(alpha))
    through = torch.cumprod(1 - alpha, 1)
    front = torch.cat([torch.ones_like(through[:, :1]), through[:, :-1]], 1)
    weight = torch.where(through >= T_MIN, alpha * front, torch.zeros_like(alpha))
    one = torch.ones_like(q[:, :1])
    return (weight @ torch.cat([q[:, 7:10], q[:, 2:3], one], 1)).T


def _loss(maps, rgb, depth, prior):
    valid = depth > 0
    seen = valid & (maps[4] > SIL)
    loss = W_RGB * ((maps[:3] - rgb).abs() * seen).sum() + W_DEPTH * ((maps[3] - depth).abs() * seen).sum()
    loss = loss + W_VIS * ((1 - maps[4]) * valid).sum()
    return loss + W_PRIOR * ((maps[3] - prior).abs() * (seen & (prior > 0))).sum()


def _exact_view(g, cam, pose, tangent, objective=None):
    """One view: its maps (5 x pixels) and, with objective(maps of some pixels, their flat
    indices) -> scalar, the objective's value, back-propagated to g and tangent."""
    q, half = _screen(g, cam, pose, tangent)
    grad, value = torch.zeros_like(q), 0.0
    out = torch.zeros(5, cam.height * cam.width, dtype=torch.float64, device=DEV)
    flat, lo, hi = q.detach(), q.detach()[:, :2] - half, q.detach()[:, :2] + half
    for y0 in range(0, cam.height, TILE):
        y1 = min(y0 + TILE, cam.height) - 1
        row = ((lo[:, 1] <= y1) & (hi[:, 1] >= y0)).nonzero()[:, 0]
        for x0 in range(0, cam.width, TILE):
            x1 = min(x0 + TILE, cam.width) - 1
            at = row[(lo[row, 0] <= x1) & (hi[row, 0] >= x0)]
            v, u = torch.meshgrid(torch.arange(y0, y1 + 1, device=DEV), torch.arange(x0, x1 + 1, device=DEV), indexing="ij")
            px = (v * cam.width + u).reshape(-1)
            leaf = flat[at].requires_grad_(objective is not None)
            maps = _composite(leaf, u.reshape(-1).double(), v.reshape(-1).double())
            out[:, px] = maps.detach()
            if objective is not None:
                part = objective(maps, px)
                value += float(part.detach())
                if at.numel():
                    grad[at] += torch.autograd.grad(part, leaf)[0]
    if objective is not None:
        q.backward(grad)
    return out, value


def exact(case, seed):
    kind = case["kind"]
    sizes = [IMAGES[k % 3] if case["mixed"] else (case["width"], case["height"]) for k in range(case["frames"])]
    if kind not in ("map", "quality") and sum(w * h for w, h in sizes) * case["hyps"] * case["iters"] > 1_300_000:
        return None
    g, cams, poses, views = _inputs(case, seed)
    s = {"case": case, "cams": cams, "poses": poses, "views": views}
    if kind == "quality":
        return _exact_quality(_prepare_quality(s, seed))
    if kind == "map":
        return _exact_map(s, g, seed)
    g = {k: None if v is None else v.double() for k, v in g.items()}
    if kind in ("track", "upload", "frame"):
        return _exact_track(case, g, cams, poses, views)
    tangent = torch.zeros(6, dtype=torch.float64, device=DEV)
    if kind == "render":
        maps = [_exact_view(g, c, p, tangent)[0] for c, p in zip(cams, poses)]
        return {"rgb": torch.cat([m[:3].reshape(-1) for m in maps]), "depth": torch.cat([m[3] for m in maps]),
                "sil": torch.cat([m[4] for m in maps])}
    g = {k: None if v is None else v.requires_grad_(True) for k, v in g.items()}
    maps, losses, first = [], [], 0
    if kind == "autograd":
        up_rgb, up_depth, up_sil = (t.double() for t in _upstream(cams, seed))
    for c, p, (rgb, depth, prior) in zip(cams, poses, views):
        P = c.width * c.height
        if kind == "window":
            rgb, depth, prior = rgb.reshape(3, -1).double(), depth.reshape(-1).double(), prior.reshape(-1).double()
            objective = lambda m, at: _loss(m, rgb[:, at], depth[at], prior[at])
        else:
            up = torch.cat([up_rgb[3 * first:3 * (first + P)].reshape(3, P), up_depth[None, first:first + P],
                            up_sil[None, first:first + P]])
            objective = lambda m, at: (m * up[:, at]).sum()
        m, value = _exact_view(g, c, p, tangent, objective)
        maps.append(m)
        losses.append(value)
        first += P
    grads = {k: v.grad for k, v in g.items() if v is not None}
    if kind == "window":
        return {"grads": grads, "loss": torch.tensor(losses, dtype=torch.float64)}
    return {"maps": [torch.cat([m[:3].reshape(-1) for m in maps]), torch.cat([m[3] for m in maps]),
                     torch.cat([m[4] for m in maps])], "grads": grads}


def _exact_track(case, g, cams, poses, views):
    """The decoupled Adam iterations of every view: rotation about the camera centre and
    shift, each with its own moments, rates 2e-3."""
    beta1, beta2, eps, lr = 0.9, 0.999, 1e-8, 2e-3
    poses, hist = poses.clone(), []
    state = torch.zeros(len(cams), 16, dtype=torch.float64, device=DEV)
    for it in range(case["iters"]):
        losses = []
        for k, (c, (rgb, depth, prior)) in enumerate(zip(cams, views)):
            rgb, depth, prior = rgb.reshape(3, -1).double(), depth.reshape(-1).double(), prior.reshape(-1).double()
            tangent = torch.zeros(6, dtype=torch.float64, device=DEV, requires_grad=True)
            _, value = _exact_view(g, c, poses[k], tangent, lambda m, at: _loss(m, rgb[:, at], depth[at], prior[at]))
            losses.append(value)
            m = state[k, [0, 1, 2, 6, 7, 8]] * beta1 + (1 - beta1) * tangent.grad
            v = state[k, [3, 4, 5, 9, 10, 11]] * beta2 + (1 - beta2) * tangent.grad.square()
            state[k, [0, 1, 2, 6, 7, 8]], state[k, [3, 4, 5, 9, 10, 11]] = m, v
            state[k, 12:15] = torch.tensor([it + 1, beta1 ** (it + 1), beta2 ** (it + 1)], dtype=torch.float64)
            step = lr * (m / (1 - beta1 ** (it + 1))) / ((v / (1 - beta2 ** (it + 1))).sqrt() + eps)
            angle = step[:3].norm()
            a = torch.cat([torch.cos(angle / 2)[None], -torch.sin(angle / 2) * step[:3] / angle])
            q, t = poses[k, :4], poses[k, 4:]
            turned = torch.cat([(a[0] * q[0] - a[1:] @ q[1:])[None],
                                a[0] * q[1:] + q[0] * a[1:] + torch.linalg.cross(a[1:], q[1:])])
            poses[k] = torch.cat([turned / turned.norm(), _rotation(a) @ t - step[3:]])
        hist.append(losses)
    out = {"pose": poses if case["kind"] != "frame" else poses[0], "loss": torch.tensor(hist, dtype=torch.float64)}
    if case["kind"] == "upload":
        out["result"] = torch.cat([poses, out["loss"][-1][:, None].to(DEV)], 1)
    return out


def _exact_map(s, g, seed):
    g, sil, cap, grads = _map_inputs(s, g, seed)
    case, cam, pose, (rgb, depth, _) = s["case"], s["cams"][0], s["poses"][0], s["views"][0]
    n, iso = g["means"].shape[0], case["isotropic"]
    new = (depth > 0) & (sil < 0.5)
    v, u = new.nonzero().T
    d = depth[new].double()
    local = torch.stack([(u - cam.cx) / cam.fx * d, (v - cam.cy) / cam.fy * d, d], 1)
    k = d.numel()
    ls = torch.log(d / cam.fx)
    added = {"means": (local - pose[4:]) @ _rotation(pose[:4]), "log_scales": ls if iso else ls[:, None].expand(k, 3),
             "logits": torch.zeros(k, dtype=torch.float64, device=DEV), "rgb": rgb[:, new].T.double()}
    if not iso:
        added["quats"] = torch.tensor([[1.0, 0, 0, 0]], dtype=torch.float64, device=DEV).expand(k, 4)
    rate = {"means": 1e-4, "quats": 1e-3, "log_scales": 1e-3, "logits": 5e-2, "rgb": 2.5e-3}
    names = [a for a in ATTRIBUTES if g[a] is not None]
    p, m, w = {}, {}, {}
    for a in names:
        before = torch.cat([g[a].double(), added[a]])
        grad = grads[a][:n + k].double()
        m[a], w[a] = 0.1 * grad, 0.001 * grad * grad
        p[a] = before - rate[a] * grad / (grad.abs() + 1e-15)
    keep = p["logits"] >= math.log(0.005 / 0.995)
    count = int(keep.sum())

    def rows(x):
        out = torch.zeros((cap,) + x.shape[1:], dtype=torch.float64, device=DEV)
        out[:count] = x[keep]
        return out

    moments = torch.cat([rows(x[a]).reshape(-1) for x in (m, w) for a in names])
    param = {a: rows(p[a]) for a in names}
    if iso:
        param["log_scales"] = param["log_scales"][:, None]
    copy = None if case["dtype"] == "fp32" else {a: param[a] for a in names if a != "means"}
    return {"map": param, "copy": copy, "moments": moments, "count": None}


def _exact_quality(s):
    cam = s["cams"][0]
    W, H = cam.width, cam.height
    (rgb, depth), (rgb_t, depth_t) = ((t[0].double(), t[1].double()) for t in (s["img"], s["obs"]))
    e = (depth - depth_t)[depth_t > 0]
    sums = torch.stack([(rgb - rgb_t).square().sum(), e.abs().sum(), torch.tensor(float(e.numel()), dtype=torch.float64, device=DEV),
                        e.square().sum()])
    x = torch.exp(-(torch.arange(11, dtype=torch.float64, device=DEV) - 5).square() / (2 * 1.5 * 1.5))
    x = x / x.sum()
    window = (x[:, None] * x[None, :])[None, None]
    mean = lambda t: torch.nn.functional.conv2d(t, window)
    a, b = rgb.reshape(3, 1, H, W), rgb_t.reshape(3, 1, H, W)
    value = torch.ones(3, dtype=torch.float64, device=DEV)
    for k, power in enumerate((0.0448, 0.2856, 0.3001, 0.2363, 0.1333)):
        ma, mb = mean(a), mean(b)
        va, vb, vab = mean(a * a) - ma * ma, mean(b * b) - mb * mb, mean(a * b) - ma * mb
        cs = ((2 * vab + 9e-4) / (va + vb + 9e-4)).mean((1, 2, 3)).clamp_min(0)
        value = value * cs ** power
        if k == 4:
            lum = ((2 * ma * mb + 1e-4) / (ma * ma + mb * mb + 1e-4)).mean((1, 2, 3)).clamp_min(0)
            value = value * lum ** power
        a, b = torch.nn.functional.avg_pool2d(a, 2), torch.nn.functional.avg_pool2d(b, 2)
    return {"sums": sums, "ssim": torch.cat([value.mean()[None], value])}
