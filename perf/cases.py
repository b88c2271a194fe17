"""Timed workloads of the rasterizer: the calls a user of this package makes.

Every iteration of the per-keyframe optimisation renders a batch of rig
cameras, forms an L1 loss and back-propagates into the Gaussians and the camera
poses; around it run the insertion test, the inter-camera merging and the
frequency scheduler.  The listed cases are those calls at this repository's own
workload sizes (a 10k-Gaussian box, a 500k-Gaussian 1080p view, the
1M-Gaussian six-camera rig, the 30-view keyframe window, the 6M-Gaussian road),
plus the options that are used beside them: the autograd function with pose and
focal gradients, depth and alpha losses, odd image sizes, per-view subsets, the
other tile shapes, rendering without a backward.  ``draw`` spreads the same
calls over the ranges in between.

``exact`` evaluates the same definitions in binary64 with plain torch (tile by
tile, autograd for the gradients).  Only the depth order follows the
renderer's documented binary32 camera depth, because the order of two Gaussians
whose binary32 depths tie is part of the definition.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2512_08498_gb300.rasterizer import CameraView, Rasterizer, l1_loss_grad, rasterize

DEV = "cuda"
SH_C0 = 0.28209479177387814


# ----------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------

def listed():
    return [
        # the smallest optimisation step through the autograd function: one
        # 256 x 256 view of 10k Gaussians; launches, allocation and host work
        dict(name="small_autograd_step", call="autograd", scene="box", n=10_000, sh=0, layout="single", width=256,
             height=256, pose=True, focal=False),
        # a viewer's frame: one 1080p view rendered without a backward
        dict(name="hd_render", call="render", scene="frustum", n=500_000, sh=3, layout="single", width=1920,
             height=1080),
        # an optimisation step on one 1080p view, list rounds chosen automatically
        dict(name="hd_step", call="step", scene="frustum", n=500_000, sh=3, layout="single", width=1920, height=1080,
             list_prefix=0.0, no_sync=True),
        # the benchmark's step: the six-camera rig in one batched call, asynchronous
        dict(name="rig_step", call="step", scene="corridor", n=1_000_000, sh=3, layout="rig", keyframes=1, width=1600,
             height=900, list_prefix=0.0, no_sync=True),
        # joint refinement of Gaussians, rig poses and focal lengths through
        # autograd, then the rig chain; a sparser scene
        dict(name="rig_refine", call="autograd", scene="corridor", n=250_000, sh=3, layout="rig", keyframes=1,
             width=1600, height=900, pose=True, focal=True),
        # the local keyframe window: 5 keyframes x 6 cameras of uneven
        # resolution, each keyframe over its own subset of 3M Gaussians
        dict(name="window_step", call="step", scene="corridor", n=3_000_000, sh=3, layout="window", keyframes=5,
             width=1920, height=1080, list_prefix=1.0, no_sync=False),
        # the largest batch: 60 1080p views of a 300 m road with 6M Gaussians
        dict(name="road_step", call="step", scene="road", n=6_000_000, sh=3, layout="rig", keyframes=10, width=1920,
             height=1080, list_prefix=0.0, no_sync=True),
        # depth- and mask-supervised step on three odd-sized views, one over a
        # subset: degree-2 SH, a background, 32 x 8 tiles
        dict(name="ragged_depth_step", call="depth_step", scene="box", n=60_000, sh=2, layout="ragged", width=1237,
             height=701, tile="32x8"),
        # insertion test of a keyframe's six images
        dict(name="rig_insertion", call="insertion", layout="rig", keyframes=1, width=1600, height=900, sigma=1.0),
        # merging of one camera's samples with the Gaussians already built
        dict(name="rig_merge", call="merge", scene="corridor", n=1_000_000, sh=3, layout="single", width=1600,
             height=900),
        # scheduler pass over a keyframe: X(I) of ground truth, level-2 ground
        # truth and rendering of six cameras, then the decisions
        dict(name="rig_schedule", call="schedule", layout="rig", keyframes=1, width=1600, height=900, level=2),
        # a scheduler pass over few small images of awkward sizes (primes, odd levels)
        dict(name="small_schedule", call="schedule", layout="ragged", width=333, height=251, level=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["autograd", "render", "step", "step", "step", "depth_step", "insertion", "merge", "schedule"])
    case = dict(call=call)
    width = _log_int(rng, 120, 1920)
    height = max(64, int(width * rng.uniform(0.5, 0.9)))
    layout = rng.choice(["single", "rig", "rig", "window", "ragged"])
    if call in ("insertion", "schedule"):
        case.update(layout="ragged" if layout == "window" else layout, width=width, height=height)
        if case["layout"] == "rig":
            case["keyframes"] = rng.randint(1, 4)
        if call == "insertion":
            case["sigma"] = rng.choice([0.5, 1.0, 1.0, 2.0])
        else:
            case["level"] = rng.choice([1, 2, 3, 4])
        return case
    scene = rng.choice(["box", "frustum", "corridor", "corridor", "road"])
    if call == "merge":
        layout = "single"
        scene = rng.choice(["corridor", "box"])
    if layout in ("rig", "window") and scene in ("box", "frustum"):
        scene = "corridor"
    if layout == "ragged" and scene in ("corridor", "road"):
        scene = "box"
    top = {"box": 100_000, "frustum": 500_000, "corridor": 2_000_000, "road": 3_000_000}[scene]
    case.update(scene=scene, n=_log_int(rng, 2_000, top), sh=rng.choice([0, 1, 2, 3, 3, 3]), layout=layout,
                width=width, height=height)
    if layout in ("rig", "window"):
        case["keyframes"] = rng.randint(1, 4)
    if call == "step":
        case.update(list_prefix=rng.choice([0.0, 1.0]), no_sync=rng.choice([True, False]))
    if call == "autograd":
        case.update(pose=rng.choice([True, False]), focal=rng.choice([True, False]))
    if call == "depth_step":
        case.update(tile=rng.choice(["16x16", "32x8", "8x32"]))
    return case


# ----------------------------------------------------------------------------
# inputs (seeded; the distributions of this repository's workloads)
# ----------------------------------------------------------------------------

def _rot(axis, a):
    c, s = math.cos(a), math.sin(a)
    m = {"x": [[1, 0, 0], [0, c, -s], [0, s, c]], "y": [[c, 0, s], [0, 1, 0], [-s, 0, c]],
         "z": [[c, -s, 0], [s, c, 0], [0, 0, 1]]}[axis]
    return np.array(m, dtype=np.float64)


def _viewmat(r_wc, centre):
    m = np.eye(4)
    m[:3, :3] = r_wc.T
    m[:3, 3] = -r_wc.T @ np.asarray(centre, np.float64)
    return m.astype(np.float32)


def _uniform(g, shape, lo, hi):
    return torch.rand(shape, generator=g, device=DEV) * (hi - lo) + lo


def _corridor(g, n, z_half):
    """Street corridor: 40% ground, 50% two facades at x = +-8 m, 10% free."""
    kind = torch.rand(n, generator=g, device=DEV)
    x, jit = _uniform(g, n, -8.0, 8.0), _uniform(g, n, -1.0, 1.0)
    y = _uniform(g, n, -10.0, 1.6)
    z = _uniform(g, n, -z_half, z_half)
    ground, facade = kind < 0.4, (kind >= 0.4) & (kind < 0.9)
    y = torch.where(ground, 1.6 + 0.3 * jit, y)
    x = torch.where(facade, torch.sign(x) * 8.0 + 0.1 * jit, x)
    return torch.stack([x, y, z], 1).contiguous()


def _gaussians(case, g):
    n, scene = case["n"], case["scene"]
    ls = _uniform(g, (n, 3), -5.0, -1.0)
    if scene == "box":
        ls = _uniform(g, (n, 3), -4.0, -1.0)
        means = torch.stack([_uniform(g, n, -2.0, 2.0), _uniform(g, n, -2.0, 2.0), _uniform(g, n, 2.0, 10.0)], 1)
    elif scene == "frustum":
        # uniform over the image, depth log-uniform in [1, 80] m
        z = torch.exp(_uniform(g, n, 0.0, math.log(80.0)))
        aspect = case["height"] / case["width"]
        means = torch.stack([_uniform(g, n, -0.873, 0.873) * z, _uniform(g, n, -0.873, 0.873) * aspect * z, z], 1)
    else:
        means = _corridor(g, n, 30.0 if scene == "corridor" else 150.0)
        if scene == "road":
            # 5% on a sky shell of radius 500 m
            d = torch.randn(n, 3, generator=g, device=DEV)
            d = d / d.norm(dim=1, keepdim=True)
            d[:, 1] = -d[:, 1].abs()
            sky = torch.rand(n, 1, generator=g, device=DEV) < 0.05
            means = torch.where(sky, 500.0 * d, means)
            ls = torch.where(sky, _uniform(g, (n, 3), 1.0, 3.0), ls)
    q = torch.randn(n, 4, generator=g, device=DEV)
    q = q / q.norm(dim=1, keepdim=True)
    sh = torch.randn(n, (case["sh"] + 1) ** 2, 3, generator=g, device=DEV) * 0.1
    sh[:, 0] = torch.rand(n, 3, generator=g, device=DEV)
    return [means.contiguous(), ls.contiguous(), q.contiguous(), torch.randn(n, generator=g, device=DEV),
            sh.contiguous()]


def _sizes(case):
    """The (width, height) of every view."""
    w, h = case["width"], case["height"]
    if case["layout"] == "ragged":
        return [(w, h), (max(17, w // 2 + 21), max(13, h * 2 // 3 + 12)), (max(19, w // 4 + 24), max(11, h * 3 // 4 - 8))]
    if case["layout"] == "single":
        return [(w, h)]
    if case["layout"] == "window":
        s = [(w, h), (max(16, w * 5 // 6), max(16, h * 5 // 6)), (max(16, w // 2), max(16, h // 2))]
        return [s[(7 * i + i // 6) % 3] for i in range(6 * case["keyframes"])]
    return [(w, h)] * (6 * case["keyframes"])


def _views(case, seed, means=None):
    """CameraViews and, per view, the transform from its keyframe's central camera."""
    rng = np.random.default_rng(seed)
    sizes = _sizes(case)
    out, rel = [], []
    if case["layout"] in ("single", "ragged"):
        f = {"frustum": 1100.0 / 1920.0}.get(case.get("scene"), 1.0)
        for i, (w, h) in enumerate(sizes):
            vm = _viewmat(_rot("y", math.radians(4.0 * i)) @ _rot("x", math.radians(-3.0 * i)), [0.15 * i, -0.1 * i, 0.0])
            if case.get("scene") == "corridor":
                vm = _viewmat(_rot("y", math.radians(rng.uniform(-20, 20))), rng.uniform(-0.5, 0.5, 3))
            sub = None
            if i == 1 and means is not None:
                # the second view leaves out every third Gaussian
                sub = torch.arange(means.shape[0], device=DEV, dtype=torch.int32)
                sub = sub[sub % 3 != 0].contiguous()
            out.append(CameraView(w, h, f * w, f * w, w / 2.0, h / 2.0, vm, sub))
            rel.append(vm[:3].astype(np.float32))
        return out, np.stack(rel)
    step = 10.0 if case.get("scene") == "road" else 2.0
    keyframes = case["keyframes"]
    offs, eul = rng.uniform(-0.02, 0.02, (6, 3)), np.deg2rad(rng.uniform(-1.0, 1.0, (6, 3)))
    counts = np.exp(rng.uniform(math.log(200_000 / 3_000_000), 0.0, keyframes))
    counts[0] = 1.0
    for k in range(keyframes):
        centre = np.array([0.0, 0.0, (k - 0.5 * (keyframes - 1)) * step])
        central = _viewmat(np.eye(3), centre).astype(np.float64)
        sub = None
        if case["layout"] == "window" and means is not None:
            # the keyframe's Gaussians: the nearest ones to its rig centre
            nk = max(1, int(counts[k] * means.shape[0]))
            d = (means - torch.tensor(centre, device=DEV, dtype=torch.float32)).square().sum(1)
            sub = torch.sort(torch.topk(d, nk, largest=False).indices).values.to(torch.int32).contiguous()
        for c in range(6):
            w, h = sizes[6 * k + c]
            r = _rot("y", 2.0 * math.pi * c / 6) @ _rot("z", eul[c][2]) @ _rot("y", eul[c][1]) @ _rot("x", eul[c][0])
            vm = _viewmat(r, centre + offs[c])
            out.append(CameraView(w, h, w / 2.0, w / 2.0, w / 2.0, h / 2.0, vm, sub))
            rel.append((vm.astype(np.float64) @ np.linalg.inv(central))[:3].astype(np.float32))
    return out, np.stack(rel)


def _npix(case):
    return sum(w * h for w, h in _sizes(case))


def _images(case, g):
    """Ground truth (smooth shading with texture) and a blurrier rendering of
    every view, flat planar RGB."""
    gt, ren = [], []
    for w, h in _sizes(case):
        coarse = torch.rand(1, 3, max(2, h // 24), max(2, w // 24), generator=g, device=DEV)
        smooth = torch.nn.functional.interpolate(coarse, size=(h, w), mode="bilinear", align_corners=False)[0]
        detail = torch.randn(3, h, w, generator=g, device=DEV)
        strong = (torch.rand(1, h, w, generator=g, device=DEV) < 0.1).float()
        gt.append((smooth + (0.04 + 0.25 * strong) * detail).clamp(0.0, 1.0).reshape(-1))
        ren.append((smooth + 0.02 * detail).clamp(0.0, 1.0).reshape(-1))
    return torch.cat(gt), torch.cat(ren)


def _inputs(case, seed):
    """Every array of the case from the seed alone."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    inp = {}
    if "scene" in case:
        inp["params"] = _gaussians(case, g)
    means = inp["params"][0] if case["layout"] in ("window", "ragged") and "scene" in case else None
    inp["views"], inp["rel"] = _views(case, seed, means)
    npix = _npix(case)
    call = case["call"]
    if call in ("step", "autograd"):
        inp["target"] = torch.rand(3 * npix, generator=g, device=DEV)
    if call == "depth_step":
        # the upstream gradients of a photometric, a depth and a mask loss
        inp["dl"] = [torch.randn(3 * npix, generator=g, device=DEV) / (3 * npix),
                     torch.randn(npix, generator=g, device=DEV) / npix,
                     torch.randn(npix, generator=g, device=DEV) / npix]
    if call in ("insertion", "schedule", "merge"):
        inp["gt"], inp["ren"] = _images(case, g)
    if call == "insertion":
        inp["depth"] = _uniform(g, npix, 2.0, 30.0)
    if call == "schedule":
        inp["uniforms"] = torch.rand(64, generator=g, device=DEV)
    if call == "merge":
        # depth map: the nearest Gaussian in each pixel, 8 m in empty ones;
        # samples: one pixel in seven
        v = inp["views"][0]
        means = inp["params"][0]
        vm = torch.tensor(v.viewmat, device=DEV)
        p = means @ vm[:3, :3].T + vm[:3, 3]
        z = p[:, 2].clamp_min(0.2)
        px, py = (v.fx * p[:, 0] / z + v.cx).floor().long(), (v.fy * p[:, 1] / z + v.cy).floor().long()
        ok = (p[:, 2] > 0.2) & (px >= 0) & (px < v.width) & (py >= 0) & (py < v.height)
        depth = torch.full((npix,), 1e9, device=DEV)
        depth.scatter_reduce_(0, (py * v.width + px)[ok], p[:, 2][ok], "amin")
        inp["depth"] = torch.where(depth < 1e8, depth, torch.full_like(depth, 8.0)).view(v.height, v.width)
        pick = torch.rand(npix, generator=g, device=DEV).topk(max(1, npix // 7)).indices
        inp["pixels"] = torch.sort(pick).values.to(torch.int32)
        prob = _uniform(g, npix, 0.2, 1.0).view(v.height, v.width)
        inp["scale"] = inp["depth"] / (2.0 * prob.sqrt() * v.fx)
    return inp


# ----------------------------------------------------------------------------
# the measured calls
# ----------------------------------------------------------------------------

def _tile(case):
    w, h = case.get("tile", "16x16").split("x")
    return int(w), int(h)


def _bg(case):
    return (0.1, 0.2, 0.3) if case["call"] == "depth_step" else (0.0, 0.0, 0.0)


def prepare(case, seed):
    inp = _inputs(case, seed)
    call = case["call"]
    st = dict(inp, case=case)
    st["raster"] = r = Rasterizer(tile=_tile(case), sh_degree=case.get("sh", 3), bg=_bg(case), device=DEV)
    npix = _npix(case)
    if call == "autograd":
        st["params"] = [p.requires_grad_(True) for p in inp["params"]]
        nv = len(inp["views"])
        st["pose"] = torch.zeros(nv, 6, device=DEV, requires_grad=True) if case["pose"] else None
        st["focal"] = torch.zeros(nv, 2, device=DEV, requires_grad=True) if case["focal"] else None
    if call in ("render", "step", "depth_step"):
        # what a render loop keeps: the output buffers and the saved state
        st["saved"] = r.new_saved()
        st["out"] = tuple(torch.empty(k * npix, device=DEV) for k in (3, 1, 1))
    if call in ("step", "depth_step"):
        st["grads"] = tuple(torch.empty_like(p) for p in inp["params"]) + (
            torch.empty(len(inp["views"]), 6, device=DEV),)
    if call == "step":
        st["dl"], st["loss"] = torch.empty(3 * npix, device=DEV), torch.zeros(1, device=DEV)
        r.set_config(list_prefix=case["list_prefix"])
        if case["no_sync"]:
            # one synchronous forward sizes the buffers of an asynchronous loop
            r.forward(st["params"], st["views"], saved=st["saved"], out=st["out"])
            r.set_config(no_sync=True, pair_counts=False)
    if call == "insertion":
        # the keyframe's kept buffers; the index buffer takes any number of samples
        st["out"] = (torch.empty(npix, device=DEV), torch.empty(npix, device=DEV),
                     torch.full((npix,), -1, device=DEV, dtype=torch.int32))
    if call == "schedule":
        images, off = [], 0
        for w, h in _sizes(case):
            a = slice(off, off + 3 * w * h)
            images.append((inp["gt"][a], inp["ren"][a], w, h))
            off += 3 * w * h
        st["images"] = ([(gt, w, h, 1) for gt, _, w, h in images] +
                        [(gt, w, h, case["level"]) for gt, _, w, h in images] +
                        [(ren, w, h, 1) for _, ren, w, h in images])
    return st


def run(st):
    case, r, views = st["case"], st["raster"], st["views"]
    call = case["call"]
    if call == "autograd":
        leaves = st["params"] + [t for t in (st["pose"], st["focal"]) if t is not None]
        for t in leaves:
            t.grad = None
        rgb, depth, alpha = rasterize(*st["params"], views, r, pose_delta=st["pose"], focal_delta=st["focal"])
        dl, loss = l1_loss_grad(rgb.detach(), st["target"], loss=torch.empty(1, device=DEV))
        rgb.backward(dl)
        out = dict(rgb=rgb.detach(), depth=depth.detach(), alpha=alpha.detach(), loss=loss)
        out.update(zip(("means", "log_scales", "quats", "opacity_logits", "sh"), (p.grad for p in st["params"])))
        if st["pose"] is not None:
            out["pose"] = st["pose"].grad
        if st["focal"] is not None:
            out["focal"] = st["focal"].grad
        if case["layout"] == "rig" and st["pose"] is not None and st["focal"] is not None:
            nv = len(views)
            out.update(r.rig_chain(out["pose"], [i // 6 for i in range(nv)], st["rel"], nv // 6,
                                   focal_grads=out["focal"], camera_of_view=[i % 6 for i in range(nv)], n_cameras=6))
        return out
    if call in ("render", "step", "depth_step"):
        rgb, depth, alpha, saved = r.forward(st["params"], views, saved=st["saved"], out=st["out"])
        out = dict(rgb=rgb, depth=depth, alpha=alpha)
        if call == "step":
            l1_loss_grad(rgb, st["target"], st["dl"], st["loss"])
            out["loss"] = st["loss"]
            grads = r.backward(st["params"], views, saved, st["dl"], grads=st["grads"])
        elif call == "depth_step":
            grads = r.backward(st["params"], views, saved, *st["dl"], grads=st["grads"])
        if call != "render":
            out.update(zip(("means", "log_scales", "quats", "opacity_logits", "sh", "pose"), grads))
        return out
    if call == "insertion":
        p_a, scale, _, count = r.insertion(st["gt"], st["ren"], st["depth"], views, sigma=case["sigma"], out=st["out"])
        return dict(p_a=p_a, scale=scale, index=st["out"][2], count=count)
    if call == "merge":
        means, ls, _, _, sh = st["params"]
        out = r.merge(views[0], means, ls, sh, st["pixels"], st["scale"], st["depth"], st["gt"])
        # the kept Gaussians take their group's colour, the others keep theirs
        out["existing_dc"] = torch.where((out["existing_action"] == 2)[:, None], out["existing_dc"], sh[:, 0])
        return out
    x = r.dft_energy(st["images"])
    n = len(views)
    out = r.frequency_schedule(x[:n], x[2 * n:], x[n:2 * n], uniforms=st["uniforms"])
    return dict(out, x=x)


# Composited (pixel, Gaussian) pairs per pixel, as the renderer counts them:
# how many an image needs follows from the scene's opacity, not from the code.
# P n / (n + n0) with (P, n0) fitted to counts over the drawn range.
PAIRS_PER_PIXEL = {"box": (80.0, 5e3), "frustum": (65.0, 3e4), "corridor": (120.0, 2.5e5), "road": (120.0, 1.2e6)}


def work(case):
    """Bytes: each input read once, each output written once.  Flops (a fused
    multiply-add is two): per composited pair about 40 forward and 60
    backward, an FFT's 5 N log2 N, a stencil tap's 2."""
    npix, call = _npix(case), case["call"]
    n = case.get("n", 0)
    row = 4 * (11 + 3 * (case.get("sh", 0) + 1) ** 2)
    if call in ("render", "step", "autograd", "depth_step"):
        p, n0 = PAIRS_PER_PIXEL[case["scene"]]
        pairs = p * n / (n + n0) * npix
        if call == "render":
            return {"bytes": n * row + 20 * npix, "flops": 40 * pairs}
        up = 20 if call == "depth_step" else 12    # upstream gradients or targets
        return {"bytes": 2 * n * row + (20 + up) * npix, "flops": 100 * pairs}
    if call == "insertion":
        r = math.ceil(3.0 * case["sigma"])
        return {"bytes": (24 + 4 + 8) * npix, "flops": 2 * 3 * 2 * (2 * r + 1) ** 2 * npix}
    if call == "merge":
        # existing: mean, scales, colour in; action, colour out.  samples (one
        # pixel in seven): pixel, scale, depth, ground truth in; outputs
        return {"bytes": n * (24 + 12 + 16) + npix / 7.0 * (4 + 8 + 12 + 36), "flops": 40 * n}
    flops = sum(2 * 3 * 2.5 * w * h * math.log2(w * h) for w, h in _sizes(case))
    level = case["level"]
    flops += sum(3 * 2.5 * (w // level) * (h // level) * math.log2(max(2, (w // level) * (h // level)))
                 for w, h in _sizes(case))
    return {"bytes": 12 * 2 * npix, "flops": flops}


# ----------------------------------------------------------------------------
# binary64 reference
# ----------------------------------------------------------------------------

def _f32(x):
    return float(np.float32(x))


def _project(par, idx, v, pose, focal):
    """Records (u, v, conic, opacity, depth, rgb) of Gaussians idx in view v,
    differentiable in the parameters, the pose perturbation and the focal."""
    mu, ls, q, o, sh = (p[idx] for p in par)
    vm = torch.tensor(np.asarray(v.viewmat), device=DEV, dtype=torch.float64)
    R0, t0 = vm[:3, :3], vm[:3, 3]
    rho, om = pose[:3], pose[3:]
    skew = torch.stack([torch.stack([om[0] * 0, -om[2], om[1]]), torch.stack([om[2], om[0] * 0, -om[0]]),
                        torch.stack([-om[1], om[0], om[0] * 0])])
    R, t = R0 + skew @ R0, t0 + skew @ t0 + rho
    fx, fy = _f32(v.fx) + focal[0], _f32(v.fy) + focal[1]
    p = mu @ R.T + t
    x, y, z = p.unbind(1)
    s = ls.exp()
    qn = q / q.norm(dim=1, keepdim=True)
    w, a, b, c = qn.unbind(1)
    rot = torch.stack([1 - 2 * (b * b + c * c), 2 * (a * b - w * c), 2 * (a * c + w * b),
                       2 * (a * b + w * c), 1 - 2 * (a * a + c * c), 2 * (b * c - w * a),
                       2 * (a * c - w * b), 2 * (b * c + w * a), 1 - 2 * (a * a + b * b)], 1).view(-1, 3, 3)
    m = rot * s[:, None, :]
    # frustum guard: fx x~ = clamp(fx x / z, +-1.3 max(cx, W - cx)) z
    gx, gy = 1.3 * max(v.cx, v.width - v.cx), 1.3 * max(v.cy, v.height - v.cy)
    fxx, fyy = (fx * x / z).clamp(-gx, gx) * z, (fy * y / z).clamp(-gy, gy) * z
    T0 = (fx / z)[:, None] * R[0] - (fxx / (z * z))[:, None] * R[2]
    T1 = (fy / z)[:, None] * R[1] - (fyy / (z * z))[:, None] * R[2]
    a0, a1 = torch.einsum("ni,nij->nj", T0, m), torch.einsum("ni,nij->nj", T1, m)
    ca, cb, cc = (a0 * a0).sum(1) + 0.3, (a0 * a1).sum(1), (a1 * a1).sum(1) + 0.3
    det = ca * cc - cb * cb
    centre = -(R0.T @ t0)
    d = mu - centre
    d = d / d.norm(dim=1, keepdim=True)
    col = (torch.einsum("nk,nkc->nc", _sh_basis(d, sh.shape[1]), sh) + 0.5).clamp_min(0.0)
    rec = torch.stack([fx * x / z + v.cx, fy * y / z + v.cy, cc / det, -cb / det, ca / det, torch.sigmoid(o), z], 1)
    return torch.cat([rec, col], 1), (ca, cb, cc, det)


def _sh_basis(d, k):
    x, y, z = d.unbind(1)
    out = [torch.full_like(x, SH_C0)]
    if k > 1:
        c = 0.4886025119029199
        out += [-c * y, c * z, -c * x]
    if k > 4:
        c0, c1, c2 = 1.0925484305920792, 0.31539156525252005, 0.5462742152960396
        out += [c0 * x * y, -c0 * y * z, c1 * (2 * z * z - x * x - y * y), -c0 * x * z, c2 * (x * x - y * y)]
    if k > 9:
        c0, c1, c2, c3, c4 = (0.5900435899266435, 2.890611442640554, 0.4570457994644658, 0.3731763325901154,
                              1.445305721320277)
        r = 4 * z * z - x * x - y * y
        out += [-c0 * y * (3 * x * x - y * y), c1 * x * y * z, -c2 * y * r, c3 * z * (2 * z * z - 3 * x * x - 3 * y * y),
                -c2 * x * r, c4 * z * (x * x - y * y), -c0 * x * (x * x - 3 * y * y)]
    return torch.stack(out, 1)


def _depth32(means, v):
    """The renderer's binary32 camera depth (fused multiply-adds, z row)."""
    r = np.asarray(v.viewmat, np.float32)[2].astype(np.float64)
    acc = torch.full((means.shape[0],), r[3], device=DEV, dtype=torch.float64)
    for i in (2, 1, 0):
        acc = (means[:, i].double() * r[i] + acc).float().double()
    return acc.float()


def _alphas(rec, live, px, py):
    """alpha of every (entry, pixel) pair, zero where the pair is skipped."""
    dx, dy = px - rec[..., 0, None], py - rec[..., 1, None]
    p = -0.5 * (rec[..., 2, None] * dx * dx + rec[..., 4, None] * dy * dy) - rec[..., 3, None] * dx * dy
    al = (rec[..., 5, None] * p.clamp_max(0.0).exp()).clamp_max(_f32(0.99))
    return torch.where(live[..., None] & (p <= 0) & (al >= _f32(1.0 / 255.0)), al, torch.zeros_like(al))


def _weights(al, T, done):
    """Blend weights of a segment of entries given the transmittance before it."""
    om = 1.0 - al
    incl = T[:, None] * torch.cumprod(om, 1)
    stop = ((al > 0) & (incl.detach() < _f32(1e-4))).cumsum(1) > 0
    alive = ~(stop | done[:, None])
    wgt = torch.where(alive, al * incl / om, torch.zeros_like(al))
    return wgt, alive, om, done | stop[:, -1]


def _tile_lists(rec, cov, z32, v, tile):
    """Per tile of the view: (start, length) into entries, in depth order."""
    ca, cb, cc, det = cov
    tw, th = tile
    tx, ty = -(-v.width // tw), -(-v.height // th)
    mid = 0.5 * (ca + cc)
    rad = (3.0 * (mid + (mid * mid - det).clamp_min(0.1).sqrt()).sqrt()).ceil()
    x0 = ((rec[:, 0] - rad) / tw).clamp(0, tx).long()
    x1 = ((rec[:, 0] + rad + tw - 1) / tw).clamp(0, tx).long()
    y0 = ((rec[:, 1] - rad) / th).clamp(0, ty).long()
    y1 = ((rec[:, 1] + rad + th - 1) / th).clamp(0, ty).long()
    cnt = ((x1 - x0) * (y1 - y0)).clamp_min(0) * (det > 0)
    order = torch.sort(z32, stable=True).indices
    order = order[cnt[order] > 0]
    e = torch.repeat_interleave(order, cnt[order])
    k = torch.arange(e.shape[0], device=DEV) - torch.repeat_interleave(cnt[order].cumsum(0) - cnt[order], cnt[order])
    wdt = (x1 - x0)[e]
    ids = ((y0[e] + k // wdt) * tx + x0[e] + k % wdt).to(torch.int32)
    del k, wdt
    perm = torch.sort(ids, stable=True).indices
    length = torch.bincount(ids, minlength=tx * ty)
    return e[perm], length.cumsum(0) - length, length, tx


def _chunks(need, budget):
    """Tiles by list length, in groups whose padded size stays under budget."""
    order = torch.argsort(need)
    lens = need[order].tolist()
    i = 0
    while i < len(lens):
        j = i + 1
        while j < len(lens) and (j + 1 - i) * max(1, lens[j]) <= budget:
            j += 1
        yield order[i:j], max(1, lens[j - 1])
        i = j


def _raster64(case, inp, want_pose=False, want_focal=False):
    """Images and, where the case has them, gradients in binary64."""
    grads = case["call"] != "render"
    tile, bg = _tile(case), torch.tensor([_f32(b) for b in _bg(case)], device=DEV, dtype=torch.float64)
    par = [p.detach().double().requires_grad_(grads) for p in inp["params"]]
    nv = len(inp["views"])
    pose = torch.zeros(nv, 6, device=DEV, dtype=torch.float64, requires_grad=grads)
    focal = torch.zeros(nv, 2, device=DEV, dtype=torch.float64, requires_grad=grads)
    npix = _npix(case)
    rgbs, depths, alphas = [], [], []
    loss = torch.zeros((), device=DEV, dtype=torch.float64)
    off = 0
    for i, v in enumerate(inp["views"]):
        hw = v.width * v.height
        with torch.no_grad():
            idx = torch.arange(par[0].shape[0], device=DEV) if v.subset is None else v.subset.long()
            z32 = _depth32(inp["params"][0][idx], v)
            idx, z32 = idx[z32 > _f32(0.2)], z32[z32 > _f32(0.2)]
            rec, cov = _project(par, idx, v, pose[i].detach(), focal[i].detach())
            entries, start, length, tx = _tile_lists(rec, cov, z32, v, tile)
            used = torch.unique(entries)
            local = torch.full((idx.shape[0],), -1, device=DEV, dtype=torch.long)
            local[used] = torch.arange(used.shape[0], device=DEV)
            entries, idx, rec = local[entries], idx[used], rec[used]
            pix = torch.arange(tile[0] * tile[1], device=DEV)
            lx, ly = pix % tile[0], pix // tile[0]

        def gather(tiles, s, e):
            pos = torch.arange(s, e, device=DEV)
            live = pos < length[tiles][:, None]
            ent = entries[(start[tiles][:, None] + pos).clamp_max(max(entries.shape[0] - 1, 0))] if len(entries) else \
                torch.zeros(live.shape, device=DEV, dtype=torch.long)
            x, y = (tiles % tx)[:, None] * tile[0] + lx, (tiles // tx)[:, None] * tile[1] + ly
            return torch.where(live, ent, torch.zeros_like(ent)), live, x, y

        # images: every tile's list in segments until all of its pixels stop
        rgb = torch.zeros(3, hw, device=DEV, dtype=torch.float64)
        dep = torch.zeros(hw, device=DEV, dtype=torch.float64)
        tfin = torch.ones(hw, device=DEV, dtype=torch.float64)
        need = torch.zeros_like(length)
        with torch.no_grad():
            for tiles in torch.argsort(length).split(512):
                _, _, x, y = gather(tiles, 0, 1)
                inside = (x < v.width) & (y < v.height)
                T = torch.ones(x.shape, device=DEV, dtype=torch.float64)
                done, acc = ~inside, torch.zeros(4, *x.shape, device=DEV, dtype=torch.float64)
                top, s = int(length[tiles].max()), 0
                while s < top and not bool(done.all()) and rec.shape[0] > 0:
                    e = min(top, s + 96)
                    ent, live, _, _ = gather(tiles, s, e)
                    need[tiles] = torch.where(done.all(1), need[tiles], torch.full_like(need[tiles], e))
                    r = rec[ent]
                    al = _alphas(r, live, x[:, None] + 0.5, y[:, None] + 0.5)
                    wgt, alive, om, done = _weights(al, T, done)
                    T = T * torch.where(alive, om, torch.ones_like(om)).prod(1)
                    for ch, col in enumerate((7, 8, 9, 6)):
                        acc[ch] += (wgt * r[..., col, None]).sum(1)
                    s = e
                at = (y * v.width + x)[inside]
                for ch in range(3):
                    rgb[ch, at] = (acc[ch] + T * bg[ch])[inside]
                dep[at], tfin[at] = acc[3][inside], T[inside]
            need = torch.minimum(need, length)
        rgbs.append(rgb.reshape(-1))
        depths.append(dep)
        alphas.append(1.0 - tfin)
        if grads:
            if case["call"] == "depth_step":
                dr = inp["dl"][0][3 * off:3 * off + 3 * hw].double().view(3, hw)
                dd, da = (t[off:off + hw].double() for t in inp["dl"][1:])
            else:
                diff = rgb - inp["target"][3 * off:3 * off + 3 * hw].double().view(3, hw)
                loss += diff.abs().sum() / (3 * npix)
                dr, dd, da = diff.sign() / (3 * npix), torch.zeros_like(dep), torch.zeros_like(dep)
            grec = torch.zeros_like(rec)
            for tiles, top in _chunks(need, 49152):
                if rec.shape[0] == 0 or top == 0:
                    continue
                ent, live, x, y = gather(tiles, 0, top)
                inside = (x < v.width) & (y < v.height)
                at = (y * v.width + x).clamp_max(hw - 1)
                up = [torch.where(inside, t[at], torch.zeros_like(dep[:1])) for t in (dr[0], dr[1], dr[2], dd, da)]
                r = rec[ent].requires_grad_(True)
                al = _alphas(r, live, x[:, None] + 0.5, y[:, None] + 0.5)
                T = torch.ones(x.shape, device=DEV, dtype=torch.float64)
                wgt, alive, om, _ = _weights(al, T, ~inside)
                tf = torch.where(alive, om, torch.ones_like(om)).prod(1)
                per = sum(u[:, None] * r[..., col, None] for u, col in zip(up, (7, 8, 9, 6)))
                out = (wgt * per).sum() + (tf * (up[0] * bg[0] + up[1] * bg[1] + up[2] * bg[2] - up[4])).sum()
                g, = torch.autograd.grad(out, r)
                grec.index_add_(0, ent.reshape(-1), g.reshape(-1, g.shape[-1]))
            if rec.shape[0] > 0:
                full, _ = _project(par, idx, v, pose[i], focal[i])
                full.backward(grec)
        off += hw
    out = dict(rgb=torch.cat(rgbs), depth=torch.cat(depths), alpha=torch.cat(alphas))
    if grads:
        if case["call"] != "depth_step":
            out["loss"] = loss.reshape(1)
        zero = lambda p: p.grad if p.grad is not None else torch.zeros_like(p)
        out.update(zip(("means", "log_scales", "quats", "opacity_logits", "sh"), map(zero, par)))
        if want_pose:
            out["pose"] = zero(pose)
        if want_focal:
            out["focal"] = zero(focal)
    return out


def _rig_chain64(pose, focal, rel):
    """Central pose (Ad(A)^T of each view's gradient), relative transforms and focals."""
    nv = pose.shape[0]
    A = torch.tensor(rel, device=DEV, dtype=torch.float64)
    rho, om = pose[:, :3], pose[:, 3:]
    w = om - torch.cross(A[:, :, 3], rho, dim=1)
    c = torch.cat([torch.einsum("vij,vi->vj", A[:, :, :3], rho), torch.einsum("vij,vi->vj", A[:, :, :3], w)], 1)
    return dict(central=c.view(nv // 6, 6, 6).sum(1), camera_rel=pose.view(nv // 6, 6, 6).sum(0),
                camera_focal=focal.view(nv // 6, 6, 2).sum(0))


def _log_response(img, w, h, sigma):
    """P(I): the clamped norm of the zero-mean LoG response."""
    r = math.ceil(3.0 * sigma)
    ax = torch.arange(-r, r + 1, device=DEV, dtype=torch.float64)
    q = ax[:, None] ** 2 + ax[None, :] ** 2
    s2 = sigma * sigma
    k = (q - 2 * s2) / (s2 * s2) * torch.exp(-q / (2 * s2)) / (2 * math.pi * s2)
    k = k - k.mean()
    pad = torch.nn.functional.pad(img.double().view(1, 3, h, w), (r, r, r, r), mode="replicate")[0]
    acc = torch.zeros(3, h, w, device=DEV, dtype=torch.float64)
    for dy in range(2 * r + 1):
        for dx in range(2 * r + 1):
            acc += k[dy, dx] * pad[:, dy:dy + h, dx:dx + w]
    return acc.square().sum(0).sqrt().clamp_max(1.0).reshape(-1)


def _merge64(inp):
    v = inp["views"][0]
    means, ls, _, _, sh = (p.double() for p in inp["params"])
    w, hw = v.width, v.width * v.height
    vm = torch.tensor(np.asarray(v.viewmat), device=DEV, dtype=torch.float64)
    R, t = vm[:3, :3], vm[:3, 3]
    x, y, z = (means @ R.T + t).unbind(1)
    u, vv = v.fx * x / z + v.cx, v.fy * y / z + v.cy
    ok = (z > _f32(0.2)) & (u >= 0) & (u < v.width) & (vv >= 0) & (vv < v.height)
    pixels = inp["pixels"].long()
    m = pixels.shape[0]
    slot_map = torch.full((hw,), -1, device=DEV, dtype=torch.long)
    slot_map[pixels] = torch.arange(m, device=DEV)
    depth, scale = inp["depth"].double().view(-1), inp["scale"].double().view(-1)
    pix = torch.where(ok, vv.floor() * w + u.floor(), torch.zeros_like(u)).long()
    ok &= (slot_map[pix] >= 0) & ((z - depth[pix]).abs() <= 0.5)
    g = ok.nonzero().flatten()
    s = slot_map[pix[g]]
    sc = ls.max(1).values.exp()[g] * v.fx / z[g]
    best = torch.full((m,), float("inf"), device=DEV, dtype=torch.float64).scatter_reduce(0, s, sc, "amin")
    cnt = torch.zeros(m, device=DEV, dtype=torch.float64).index_add(0, s, torch.ones_like(sc))
    d = depth[pixels]
    dc = ((inp["gt"].double().view(3, hw)[:, pixels] - 0.5) / SH_C0).T
    mean_dc = (dc + torch.zeros_like(dc).index_add(0, s, sh[g, 0])) / (cnt + 1)[:, None]
    mean_d = (d + torch.zeros_like(d).index_add(0, s, z[g])) / (cnt + 1)
    replaces = (cnt > 0) & (scale[pixels] * v.fx / d < best)
    dep = torch.where(replaces, mean_d, d)
    px, py = (pixels % w).double() + 0.5, (pixels // w).double() + 0.5
    cam = torch.stack([(px - v.cx) / v.fx * dep, (py - v.cy) / v.fy * dep, dep], 1)
    win = g[(sc == best[s]) & ~replaces[s]]
    edc = sh[:, 0].clone()
    edc[win] = mean_dc[slot_map[pix[win]]]
    return dict(sample_action=None, sample_means=(cam - t) @ R, sample_scale=scale[pixels] * dep / d, sample_depth=dep,
                sample_dc=torch.where(replaces[:, None], mean_dc, dc), existing_action=None, existing_dc=edc)


def exact(case, seed):
    call = case["call"]
    if call in ("render", "step", "autograd", "depth_step"):
        # the tile-by-tile evaluation takes minutes on the largest batches
        if _npix(case) > 9_000_000 or case["n"] * len(_sizes(case)) > 6_500_000:
            return None
    inp = _inputs(case, seed)
    if call in ("render", "step", "depth_step"):
        return _raster64(case, inp, want_pose=call != "render")
    if call == "autograd":
        both = case["layout"] == "rig" and case["pose"] and case["focal"]
        out = _raster64(case, inp, want_pose=case["pose"], want_focal=case["focal"])
        if both:
            out.update(_rig_chain64(out["pose"], out["focal"], inp["rel"]))
        return out
    if call == "merge":
        return _merge64(inp)
    if call == "insertion":
        p_a, scale, off = [], [], 0
        for v in inp["views"]:
            hw = v.width * v.height
            a = slice(3 * off, 3 * (off + hw))
            pi = _log_response(inp["gt"][a], v.width, v.height, case["sigma"])
            pr = _log_response(inp["ren"][a], v.width, v.height, case["sigma"])
            pa = (pi - pr).clamp_min(0.0)
            s = inp["depth"][off:off + hw].double() / (2.0 * pi.clamp_min(1e-300).sqrt() * v.fx)
            p_a.append(pa)
            scale.append(torch.where(pa > _f32(0.2), s, torch.zeros_like(s)))
            off += hw
        return dict(p_a=torch.cat(p_a), scale=torch.cat(scale), index=None, count=None)
    xs, off = {0: [], 1: [], 2: []}, 0
    for w, h in _sizes(case):
        a = slice(off, off + 3 * w * h)
        for k, (src, f) in enumerate(((inp["gt"], 1), (inp["gt"], case["level"]), (inp["ren"], 1))):
            img = src[a].double().view(3, h, w)[:, :h // f * f, :w // f * f]
            img = img.reshape(3, h // f, f, w // f, f).mean((2, 4))
            xs[k].append(torch.fft.fft2(img).abs().square().sum(0).sqrt().sum())
        off += 3 * w * h
    xg, xl, xr = (torch.stack(xs[k]) for k in range(3))
    return dict(r=xg / xr, r_level=xl / xr, level_up=None, samples=None, x=torch.cat([xg, xl, xr]))
