"""The workloads this renderer's speed is measured on.

Every case is one call of a public entry point (paper_2609_30741_gb300.gs) on inputs a user's program has in hand:
a scene resident on the GPU, head poses, images, feature stacks. Sizes are those of the repository's own workloads
(synth.py, bench.py, the tests), widened to odd and ragged ones; scenes follow synth.py's distributions but are drawn
on the GPU. Rasterizer configurations are the context's default, or the ones the autotuner settles on at these sizes.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2609_30741_gb300 import gs, repair_train, synth

TUNED = (32, 2, 128)      # full frames of the large scenes
TUNED_ROI = (16, 2, 128)  # their ROI re-render


def listed():
    return [
        # the smallest frame: a preview or a test scene, where launches and latency count
        {"name": "stereo_small", "call": "stereo", "scene": "slab", "n": 20000, "sh": 0, "w": 256, "h": 192, "f": 300.0},
        # the headline: an object capture for a desktop stereo display
        {"name": "stereo_object", "call": "stereo", "scene": "object", "n": 500000, "sh": 3, "w": 1600, "h": 1200,
         "f": 1600.0, "tuned": True},
        # an unbounded capture at 1080p with the learned hole repair
        {"name": "stereo_unbounded_learned", "call": "stereo", "scene": "unbounded", "n": 1500000, "sh": 3, "w": 1920,
         "h": 1080, "f": 1600.0, "tuned": True, "repair": 1},
        # one headset frame (both eyes of a 2448 x 2448 panel)
        {"name": "stereo_headset", "call": "stereo", "scene": "unbounded", "n": 3000000, "sh": 3, "w": 2448, "h": 2448,
         "f": 1800.0, "tuned": True},
        # a single view of a 3DGS (ellipsoid) scene in a window of odd size, over a background colour
        {"name": "mono_ellipsoids", "call": "mono", "scene": "object", "n": 300000, "sh": 2, "w": 1237, "h": 823,
         "f": 1250.0, "ellipsoids": True},
        # the sequential two-eye render, eyes converging (toed in), ragged size
        {"name": "two_pass_toed_in", "call": "two_pass", "scene": "slab", "n": 200000, "sh": 1, "w": 1001, "h": 751,
         "f": 1170.0, "toe": 1.5},
        # serving: eight stereo frames of four scenes of different sizes in one call (the largest)
        {"name": "batch_serving", "call": "batch", "n": 4900000, "sh": 3, "w": 2048, "poses": 2},
        # the repair network alone on the hole tiles of a frame, BF16 and FP8
        {"name": "repair_bf16", "call": "infer", "tiles": 1000, "frames": 1, "w": 1920, "h": 1080, "fp8": 0},
        {"name": "repair_fp8", "call": "infer", "tiles": 2600, "frames": 3, "w": 1601, "h": 1203, "fp8": 1},
        # one training step of the repair network (the trainer's batch)
        {"name": "repair_train", "call": "train", "tiles": 512, "frames": 2, "w": 1600, "h": 1200},
        # quality metric of a rendered frame
        {"name": "ssim", "call": "ssim", "w": 1919, "h": 1079, "c": 3},
        # the allocation-free warp a compositor calls
        {"name": "warp_noalloc", "call": "warp", "w": 1600, "h": 1200, "f": 1600.0},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["stereo", "stereo", "stereo", "mono", "mono", "two_pass", "batch", "infer", "train", "ssim",
                       "warp"])
    if call in ("stereo", "mono", "two_pass"):
        scene = rng.choice(["slab", "object", "unbounded"])
        n = _log(rng, 10000, {"slab": 400000, "object": 1200000, "unbounded": 3000000}[scene])
        w = _log(rng, 250, 2448 if scene == "unbounded" else 1920)
        if scene != "unbounded":  # near surfels grow with the image: no more of them than the object frame has
            n = min(n, int(500000 * (1600 / w) ** 2))
        h = max(160, min(2448, int(w * rng.uniform(0.55, 1.0))))
        fov = {"slab": 1.17, "object": 1.0, "unbounded": 0.75}[scene]
        c = {"call": call, "scene": scene, "n": n, "sh": rng.randrange(4), "w": w, "h": h, "f": round(w * fov, 1)}
        if rng.random() < 0.4:
            c["ellipsoids"] = True
        if rng.random() < 0.5 and w >= 600:
            c["tuned"] = True
        if call != "mono" and rng.random() < 0.3:
            c["toe"] = round(rng.uniform(0.5, 2.0), 2)
        if call == "stereo" and scene == "unbounded" and rng.random() < 0.4:
            c["repair"] = 1
        return c
    if call == "batch":
        return {"call": "batch", "n": _log(rng, 200000, 4800000), "sh": rng.randrange(4), "w": _log(rng, 500, 2047),
                "poses": rng.randrange(1, 3)}
    w, h = _log(rng, 500, 2047), _log(rng, 400, 2047)
    if call == "infer":
        frames = rng.randrange(1, 4)
        return {"call": "infer", "tiles": min(_log(rng, 60, 6000), frames * (w // 16) * (h // 16)), "frames": frames,
                "w": w, "h": h, "fp8": rng.randrange(2)}
    if call == "train":
        return {"call": "train", "tiles": _log(rng, 100, 600), "frames": rng.randrange(1, 4), "w": w, "h": h}
    if call == "ssim":
        return {"call": "ssim", "w": w, "h": h, "c": rng.choice([1, 3])}
    return {"call": "warp", "w": w, "h": h, "f": float(w)}


# ------------------------------------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _uniform(g, lo, hi, *shape):
    return torch.rand(*shape, generator=g, device="cuda") * (hi - lo) + lo


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _ball(g, n, radius, centre):
    d = _normal(g, n, 3)
    d = d / d.norm(dim=1, keepdim=True)
    return d * (radius * _uniform(g, 0, 1, n, 1) ** (1 / 3)) + torch.tensor(centre, device="cuda")


def _scene(g, kind, n, sh, ellipsoids=False):
    """synth.py's slab + ball, object + ground and unbounded distributions, drawn on the GPU."""
    scale = torch.exp(math.log(0.02) + 0.5 * _normal(g, n, 2))
    quat = _normal(g, n, 4)
    quat = quat / quat.norm(dim=1, keepdim=True)
    k = (sh + 1) ** 2
    coeff = 0.2 * _normal(g, n, k, 3)
    if kind == "slab":
        nf = n // 5
        nb = n - nf
        lo, hi = torch.tensor([-2.0, -1.5, 3.0], device="cuda"), torch.tensor([2.0, 1.5, 4.0], device="cuda")
        xyz = torch.cat([torch.rand(nb, 3, generator=g, device="cuda") * (hi - lo) + lo, _ball(g, nf, 0.5, (0.0, 0.0, 1.5))])
        coeff[:, 0] = _uniform(g, -math.sqrt(math.pi), math.sqrt(math.pi), n, 3)
    elif kind == "object":
        ng = n // 10
        nc = n - ng
        ground = torch.stack([_uniform(g, -2, 2, ng), torch.full((ng,), 0.6, device="cuda"), _uniform(g, 0.5, 4, ng)], 1)
        xyz = torch.cat([0.3 * _normal(g, nc, 3) + torch.tensor([0.0, 0.0, 2.0], device="cuda"), ground])
        phi = _uniform(g, 0, 2 * math.pi, ng) / 2  # ground surfels face up
        s = math.sqrt(0.5)
        quat[nc:] = torch.stack([s * phi.cos(), -s * phi.cos(), s * phi.sin(), s * phi.sin()], 1)
    else:
        ns = int(round(0.4 * n))
        d = _normal(g, ns, 3)
        d = d / d.norm(dim=1, keepdim=True)
        xyz = torch.cat([_ball(g, n - ns, 1.0, (0.0, 0.0, 0.0)), d * _uniform(g, 10, 30, ns, 1)])
        scale[n - ns:] = torch.exp(_uniform(g, math.log(0.03), math.log(0.3), ns, 2))
    if ellipsoids:  # a third axis along the normal, thinner than the others
        scale = torch.cat([scale, 0.3 * scale.amin(1, keepdim=True), torch.zeros(n, 1, device="cuda")], 1)
    pos = torch.cat([xyz, torch.zeros(n, 1, device="cuda")], 1)
    return synth.Scene(pos.contiguous(), quat.contiguous(), scale.contiguous(), _uniform(g, 0.3, 0.99, n),
                       coeff.contiguous(), sh, 1 if ellipsoids else 0)


def _head(seed, kind, toe=0.0):
    """A head pose looking at the scene and its two eyes 64 mm apart; toe: degrees each eye turns inwards."""
    r = np.random.RandomState(int(seed) % (1 << 31))
    yaw = math.radians(r.uniform(-15, 15))
    if kind == "slab":
        head = synth.look_at((r.uniform(-0.1, 0.1), r.uniform(-0.05, 0.05), 0.0), (0.0, 0.0, 3.5))
    else:
        radius, centre = (2.0, (0.0, 0.0, 2.0)) if kind == "object" else (3.0, (0.0, 0.0, 0.0))
        head = synth.look_at(np.array(centre) + radius * np.array([math.sin(yaw), 0.0, -math.cos(yaw)]), centre)
    dom, aff = synth.eye_pair(head)
    if toe:
        def turned(p, a):
            c, s = math.cos(a), math.sin(a)
            return synth.Pose(p.R @ np.array([[c, 0.0, s], [0.0, 1.0, 0.0], [-s, 0.0, c]]), p.t)
        dom, aff = turned(dom, math.radians(toe)), turned(aff, math.radians(-toe))
    return dom, aff


def _context(n, w, h, paths=0):
    # room for the (surfel, tile) pairs of views that fill the image with surfels some 50 pixels wide
    room = max(1 << 21, min(1 << 27, 96 * n))
    return gs.Context(n, w, h, max_instances=room, paths=paths)


def _outputs(ctx, cam):
    out = ctx.alloc_outputs(cam)
    out["roi_rects"].zero_()  # only the rectangles found are written
    out["cls_aff"].zero_()
    return out


def _batch_scenes(case):
    """(kind, surfels, width, height, focal length) of the batch's four scenes, sized by the case."""
    s, k = case["n"] / 4.9e6, case["w"] / 2048
    size = lambda v: max(96, int(round(v * k)))
    return [("slab", max(4000, int(0.2e6 * s)), size(1280), size(720), 1500.0 * k),
            ("object", max(4000, int(0.5e6 * s)), size(1600), size(1200), 1600.0 * k),
            ("object", max(4000, int(1.2e6 * s)), size(1920), size(1080), 1920.0 * k),
            ("unbounded", max(4000, int(3.0e6 * s)), size(2048), size(1536), 1506.0 * k)]


def _smooth(g, c, h, w, cell=48):
    z = torch.rand(1, c, h // cell + 2, w // cell + 2, generator=g, device="cuda")
    return torch.nn.functional.interpolate(z, size=(h, w), mode="bicubic", align_corners=False)[0].clamp(0, 1).contiguous()


def _discs(g, h, w, count):
    """Index of the topmost of `count` random discs at every pixel (-1: none)."""
    top = torch.full((h, w), -1, dtype=torch.int64, device="cuda")
    y, x = torch.arange(h, device="cuda").view(h, 1), torch.arange(w, device="cuda").view(1, w)
    p = torch.rand(count, 3, generator=g, device="cuda").cpu().tolist()
    for i, (a, b, r) in enumerate(p):
        rad = (0.02 + 0.12 * r) * w
        top[(x - a * w) ** 2 + (y - b * h) ** 2 < rad * rad] = i
    return top


def _features(g, frames, h, w):
    """Repair-network inputs of warped frames: colour, inverse depth, hole mask, distance to the nearest hole."""
    feat = torch.zeros(frames, h, w, 8, dtype=torch.bfloat16, device="cuda")
    for f in range(frames):
        top = _discs(g, h, w, 60)
        hole = torch.zeros(h, w, dtype=torch.bool, device="cuda")  # disocclusions trail the discs' right edges
        width = 3 + f
        hole[:, width:] = (top[:, :-width] >= 0) & (top[:, width:] != top[:, :-width])
        hole |= torch.rand(h, w, generator=g, device="cuda") < 0.0015
        dist = torch.full((h, w), 8.0, device="cuda")
        grown = hole.float()[None, None]
        for d in range(8):
            dist = torch.where((grown[0, 0] > 0) & (dist > d), torch.full_like(dist, float(d)), dist)
            grown = torch.nn.functional.max_pool2d(grown, 3, 1, 1)
        depth = 0.25 + 0.5 * torch.rand(61, generator=g, device="cuda")[top + 1]
        feat[f, :, :, :3] = _smooth(g, 3, h, w).permute(1, 2, 0).to(torch.bfloat16)
        feat[f, :, :, 3] = torch.where(hole, torch.zeros_like(depth), depth).to(torch.bfloat16)
        feat[f, :, :, 4] = hole.to(torch.bfloat16)
        feat[f, :, :, 5] = (dist / 8).to(torch.bfloat16)
    return feat


def _tiles(g, feat, count):
    """`count` 16 x 16 tiles (frame << 24 | y << 12 | x), those with holes first."""
    hole = feat[:, :, :, 4].float()[:, None]
    has = torch.nn.functional.max_pool2d(hole, 16, 16, ceil_mode=True)[:, 0].flatten()
    tx, ty = -(-feat.shape[2] // 16), -(-feat.shape[1] // 16)
    order = torch.argsort(-has + 0.5 * torch.rand(has.numel(), generator=g, device="cuda"))
    pick = order[torch.arange(count, device="cuda") % order.numel()]
    f, r = pick // (tx * ty), pick % (tx * ty)
    return ((f << 24) | ((r // tx) << 12) | (r % tx)).to(torch.int32)


def _weights(g):
    """The packaged network, each parameter moved a little by the seed (a network in training)."""
    w = torch.from_numpy(np.load(repair_train.UNBOUNDED_WEIGHTS).astype(np.float32).ravel()).cuda()
    return (w * (1 + 0.01 * _normal(g, w.numel()))).cpu().numpy()


ADAM = dict(lr=1e-3, beta1=0.9, beta2=0.999, eps=1e-8, weight_decay=1e-4, gate_weight=1.0)
STEPS = 200  # optimiser steps behind the training case's state


def _train_inputs(case, g):
    feat = _features(g, case["frames"], case["h"], case["w"])
    rgb = feat[..., :3].float().permute(0, 3, 1, 2)
    noise = lambda s: s * _normal(g, *rgb.shape)
    target = (rgb + noise(0.05)).clamp(0, 1).contiguous()
    plain = (rgb + noise(0.03)).clamp(0, 1).contiguous()
    w = _weights(g)
    m = (1e-4 * _normal(g, w.size)).cpu().numpy()
    v = ((1e-3 * _normal(g, w.size)) ** 2 + 1e-8).cpu().numpy()
    return feat, target, plain, _tiles(g, feat, case["tiles"]), w, m, v


def _warp_inputs(case, g):
    h, w = case["h"], case["w"]
    top = _discs(g, h, w, 40)
    depth = 1.0 + 2.0 * torch.rand(41, generator=g, device="cuda")[top + 1] + 0.05 * _smooth(g, 1, h, w)[0]
    trans = torch.where(_smooth(g, 1, h, w, 160)[0] < 0.25, torch.ones_like(depth), 0.02 * torch.rand(h, w, generator=g, device="cuda"))
    return _smooth(g, 3, h, w), (depth * (1 - trans)).contiguous(), trans.contiguous()


def prepare(case, seed):
    g = _gen(seed)
    call = case["call"]
    s = {"case": case}
    if call in ("stereo", "mono", "two_pass"):
        s["scene"] = gs.DeviceScene(_scene(g, case["scene"], case["n"], case["sh"], case.get("ellipsoids", False)))
        s["cam"] = synth.centred_camera(case["w"], case["h"], case["f"])
        s["eyes"] = _head(seed, case["scene"], case.get("toe", 0.0))
        paths = {"stereo": gs.PATH_STEREO | (gs.PATH_REPAIR if case.get("repair") else 0)}.get(call, gs.PATH_MONO)
        ctx = s["ctx"] = _context(case["n"], case["w"], case["h"], paths)
        if case.get("tuned"):
            ctx.set_raster(*TUNED)
            ctx.set_raster_roi(TUNED_ROI)
        if call == "mono":
            h, w = case["h"], case["w"]
            s["bg"] = (0.2, 0.3, 0.4)
            s["out"] = tuple(torch.zeros(shape, device="cuda") for shape in ((3, h, w), (h, w), (h, w)))
        else:
            s["out"] = _outputs(ctx, s["cam"]) if call == "stereo" else ctx.alloc_outputs(s["cam"], with_cls=False)
        if case.get("repair"):
            ctx.repair_load(np.load(repair_train.UNBOUNDED_WEIGHTS))
        s["roi"] = gs.roi_params(repair_mode=case.get("repair", 0))
    elif call == "batch":
        s["ctxs"], s["frames"], k = [], [], 0
        for kind, n, w, h, f in _batch_scenes(case):
            ds, cam = gs.DeviceScene(_scene(g, kind, n, case["sh"])), synth.centred_camera(w, h, f)
            for p in range(case["poses"]):
                ctx = _context(n, w, h, gs.PATH_STEREO)
                dom, aff = _head(seed + 7 * k + p, kind)
                s["ctxs"].append(ctx)
                s["frames"].append((ds, dom, aff, cam, _outputs(ctx, cam)))
            k += 1
        s["batch"] = gs.Batch(s["ctxs"])
        s["batch"].set_raster(*TUNED)
    elif call in ("infer", "train"):
        ctx = s["ctx"] = gs.Context(1024, case["w"], case["h"], max_instances=1 << 12, paths=gs.PATH_REPAIR)
        if call == "train":
            s["feat"], s["target"], s["plain"], s["tiles"], w, m, v = _train_inputs(case, g)
            ctx.repair_load_state(w, m, v, STEPS)
            s["scratch"] = ctx.repair_scratch(case["tiles"])
        else:
            s["feat"] = _features(g, case["frames"], case["h"], case["w"])
            s["tiles"] = _tiles(g, s["feat"], case["tiles"])
            ctx.repair_load(_weights(g))
            if case["fp8"]:
                ctx.repair_calibrate_fp8(s["feat"], s["tiles"][:64].contiguous())
            s["fill"] = torch.zeros(case["frames"], 3, case["h"], case["w"], device="cuda")
            s["gate"] = torch.zeros(case["tiles"], device="cuda")
    elif call == "ssim":
        s["ctx"] = gs.Context(1024, case["w"], case["h"], max_instances=1 << 12, paths=gs.PATH_MONO)
        s["img"], s["ref"] = _ssim_inputs(case, g)
        s["value"] = torch.zeros((), device="cuda")
    else:
        s["rgb"], s["depth"], s["trans"] = _warp_inputs(case, g)
        s["cam"] = synth.centred_camera(case["w"], case["h"], case["f"])
        s["eyes"] = _head(seed, "object")
        s["warped"] = torch.zeros_like(s["rgb"])
        s["warped_depth"] = torch.zeros_like(s["depth"])
        s["hole"] = torch.zeros(case["h"], case["w"], dtype=torch.uint8, device="cuda")
    return s


def _ssim_inputs(case, g):
    ref = _smooth(g, case["c"], case["h"], case["w"], 24)
    return (ref + 0.05 * _normal(g, *ref.shape)).contiguous(), ref


# ------------------------------------------------------------------------------------------------ one pass

def run(s):
    call = s["case"]["call"]
    if call == "stereo":
        return s["ctx"].render_stereo(s["scene"], *s["eyes"], s["cam"], gap_thresh=2, roi=s["roi"], out=s["out"])
    if call == "mono":
        rgb, depth, trans = s["ctx"].render_mono(s["scene"], s["eyes"][0], s["cam"], bg=s["bg"], out=s["out"])
        return {"rgb": rgb, "depth": depth, "trans": trans}
    if call == "two_pass":
        return s["ctx"].render_two_pass(s["scene"], *s["eyes"], s["cam"], out=s["out"])
    if call == "batch":
        s["batch"].render_stereo(s["frames"], gap_thresh=2)
        keep = ("rgb_dom", "depth_dom", "trans_dom", "rgb_aff", "cls_aff", "roi_rects", "roi_count")
        return [{k: f[4][k] for k in keep} for f in s["frames"]]
    if call == "infer":
        fill, gate = s["ctx"].repair_infer(s["feat"], s["tiles"], fill=s["fill"], gate=s["gate"], fp8=bool(s["case"]["fp8"]))
        return {"fill": fill, "gate": gate}
    if call == "train":
        ctx = s["ctx"]
        loss = ctx.repair_train_step(s["feat"], s["target"], s["plain"], s["tiles"], scratch=s["scratch"], **ADAM)
        return {"loss": loss, "gradients": ctx.repair_read(1), "weights": ctx.repair_read(0)}
    if call == "ssim":
        return s["ctx"].ssim(s["img"], s["ref"], out=s["value"])
    gs.warp_noalloc(s["rgb"], s["depth"], s["trans"], *s["eyes"], s["cam"], s["warped"], s["warped_depth"], s["hole"])
    return {"rgb": s["warped"], "depth": s["warped_depth"], "hole": s["hole"]}


# Contributions to a pixel before it is opaque, and the share of the affiliated eye a stereo frame re-renders, as the
# library's own pair counters give them on these scenes; a contribution is some 30 operations.
BLENDS = {"slab": 50, "object": 55, "unbounded": 58}
REDRAWN = {"slab": 0.4, "object": 0.2, "unbounded": 0.05}


def _render_work(kind, n, sh, pixels, eyes, redrawn, ellipsoids, images):
    """Scene attributes read once, images written once; per surfel and eye its projection and colour, per pixel its blends."""
    scene = 4 * n * (4 + 4 + (4 if ellipsoids else 2) + 1 + 3 * (sh + 1) ** 2)
    flops = n * eyes * (200 + 6 * (sh + 1) ** 2) + 30 * BLENDS[kind] * pixels * (1 + redrawn)
    return {"bytes": scene + images * pixels, "flops": flops}


NET_FLOPS = 2 * 9 * (6 * 32 + 4 * 32 * 32 + 32 * 4)  # per output pixel


def work(case):
    call, px = case["call"], case["w"] * case.get("h", 0)
    if call in ("stereo", "mono", "two_pass"):
        kind, n, sh, e = case["scene"], case["n"], case["sh"], case.get("ellipsoids", False)
        if call == "mono":
            return _render_work(kind, n, sh, px, 1, 0, e, 20)
        if call == "two_pass":
            return _render_work(kind, n, sh, px, 2, 1, e, 32)
        return _render_work(kind, n, sh, px, 2, REDRAWN[kind], e, 33)
    if call == "batch":
        total = {"bytes": 0, "flops": 0}
        for kind, n, w, h, _ in _batch_scenes(case):
            one = _render_work(kind, n, case["sh"], w * h, 2, REDRAWN[kind], False, 33)
            scene = one["bytes"] - 33 * w * h  # read once for all its poses
            total["bytes"] += scene + case["poses"] * 33 * w * h
            total["flops"] += case["poses"] * one["flops"]
        return total
    if call == "infer":
        t = case["tiles"]
        return {"bytes": t * (28 * 28 * 12 + 256 * 12 + 8) + 4 * gs.REPAIR_PARAMS, "flops": t * 256 * NET_FLOPS}
    if call == "train":
        t = case["tiles"]
        return {"bytes": t * (28 * 28 * 12 + 256 * 24 + 4) + 7 * 4 * gs.REPAIR_PARAMS, "flops": 3 * t * 256 * NET_FLOPS}
    if call == "ssim":
        return {"bytes": 8 * px * case["c"], "flops": px * case["c"] * (2 * 11 * 2 * 5 + 30)}
    return {"bytes": (20 + 17) * px, "flops": 40 * px}


# ------------------------------------------------------------------------------------------------ 64-bit values

def _sh_basis(d, deg):
    x, y, z = d.unbind(1)
    b = [torch.full_like(x, 0.5 / math.sqrt(math.pi))]
    if deg >= 1:
        k = math.sqrt(3 / (4 * math.pi))
        b += [-k * y, k * z, -k * x]
    if deg >= 2:
        k = math.sqrt(15 / math.pi) / 2
        b += [k * x * y, -k * y * z, math.sqrt(5 / math.pi) / 4 * (2 * z * z - x * x - y * y), -k * x * z, k / 2 * (x * x - y * y)]
    if deg >= 3:
        a, c = math.sqrt(35 / (2 * math.pi)) / 4, math.sqrt(21 / (2 * math.pi)) / 4
        e = math.sqrt(105 / math.pi) / 2
        b += [-a * y * (3 * x * x - y * y), e * x * y * z, -c * y * (4 * z * z - x * x - y * y),
              math.sqrt(7 / math.pi) / 4 * z * (2 * z * z - 3 * x * x - 3 * y * y), -c * x * (4 * z * z - x * x - y * y),
              e / 2 * z * (x * x - y * y), -a * x * (x * x - 3 * y * y)]
    return torch.stack(b, 1)


def _exact_view(sc, pose, w, h, f, bg=(0.0, 0.0, 0.0)):
    """One eye in 64 bits: front-to-back blending of every splat over the pixels of its bounds, 32 x 32 pixels at a time."""
    D = torch.float64
    P, q, s, o, sh = (t.to(D) for t in (sc.pos[:, :3], sc.quat, sc.scale, sc.opacity, sc.sh))
    R, t = torch.tensor(pose.R, dtype=D, device="cuda"), torch.tensor(pose.t, dtype=D, device="cuda")
    d = P - t
    col = (0.5 + torch.einsum("nk,nkc->nc", _sh_basis(d / d.norm(dim=1, keepdim=True), sc.sh_degree), sh)).clamp_min(0)
    c = d @ R  # camera coordinates
    q = q / q.norm(dim=1, keepdim=True)
    a, x, y, z = q.unbind(1)
    rot = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - a * z), 2 * (x * z + a * y), 2 * (x * y + a * z),
                       1 - 2 * (x * x + z * z), 2 * (y * z - a * x), 2 * (x * z - a * y), 2 * (y * z + a * x),
                       1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    axes = R.T @ rot  # columns: the splat's axes in the camera frame
    k2 = 2 * torch.log(255 * o)  # support radius squared
    zc, cx, cy = c[:, 2], (w - 1) / 2, (h - 1) / 2
    ok = zc > 0.2
    iz = 1 / zc.clamp_min(0.2)
    u0, v0 = f * c[:, 0] * iz + cx, f * c[:, 1] * iz + cy
    if sc.primitive:
        m = axes * s[:, None, :3]
        jx = f * iz[:, None] * (m[:, 0] - (c[:, 0] * iz)[:, None] * m[:, 2])
        jy = f * iz[:, None] * (m[:, 1] - (c[:, 1] * iz)[:, None] * m[:, 2])
        sxx, syy, sxy = (jx * jx).sum(1) + 0.3, (jy * jy).sum(1) + 0.3, (jx * jy).sum(1)
        det = sxx * syy - sxy * sxy
        rec = torch.stack([u0, v0, k2, zc, syy / det, -sxy / det, sxx / det], 1)
        ex, ey = (k2 * sxx).sqrt(), (k2 * syy).sqrt()
        box = torch.stack([u0 - ex, u0 + ex, v0 - ey, v0 + ey], 1)
    else:
        tu, tv = axes[:, :, 0] * s[:, :1], axes[:, :, 1] * s[:, 1:2]
        r = k2.clamp_min(0).sqrt()[:, None]
        us, vs = [], []
        for i, j in ((-1, -1), (1, -1), (-1, 1), (1, 1)):
            p = c + i * r * tu + j * r * tv
            ok = ok & (p[:, 2] > 0.2)
            us.append(f * p[:, 0] / p[:, 2].clamp_min(0.2) + cx)
            vs.append(f * p[:, 1] / p[:, 2].clamp_min(0.2) + cy)
        lp = (0.5 * k2).clamp_min(0).sqrt()
        us, vs = torch.stack(us + [u0 - lp, u0 + lp], 1), torch.stack(vs + [v0 - lp, v0 + lp], 1)
        box = torch.stack([us.amin(1), us.amax(1), vs.amin(1), vs.amax(1)], 1)
        rec = torch.cat([torch.stack([u0, v0, k2, zc], 1), tu, tv, c], 1)
    ok = ok & (255 * o >= 1) & (box[:, 1] >= 0) & (box[:, 0] <= w - 1) & (box[:, 3] >= 0) & (box[:, 2] <= h - 1)
    idx = torch.nonzero(ok)[:, 0]
    idx = idx[torch.argsort(zc[idx], stable=True)]
    rec, box, col, o = rec[idx], box[idx], col[idx], o[idx]
    rgb, dep, tr = (torch.empty(n, dtype=D, device="cuda") for n in ((3, h, w), (h, w), (h, w)))
    E = 32
    for y0 in range(0, h, E):
        row = torch.nonzero((box[:, 3] >= y0) & (box[:, 2] <= min(y0 + E, h) - 1))[:, 0]
        bx = box[row]
        for x0 in range(0, w, E):
            x1, y1 = min(x0 + E, w), min(y0 + E, h)
            sel = row[(bx[:, 1] >= x0) & (bx[:, 0] <= x1 - 1)]
            py, px = torch.meshgrid(torch.arange(y0, y1, dtype=D, device="cuda"), torch.arange(x0, x1, dtype=D, device="cuda"), indexing="ij")
            px, py = px.reshape(1, -1), py.reshape(1, -1)
            T = torch.ones(px.shape[1], dtype=D, device="cuda")
            C, Z = torch.zeros(3, px.shape[1], dtype=D, device="cuda"), torch.zeros_like(T)
            done = torch.zeros_like(T, dtype=torch.bool)
            for b in range(0, sel.numel(), 1024):
                i = sel[b:b + 1024]
                e = rec[i][:, :, None]
                dx, dy, z = px - e[:, 0], py - e[:, 1], e[:, 3].expand(-1, px.shape[1])
                if sc.primitive:
                    rho = e[:, 4] * dx * dx + 2 * e[:, 5] * dx * dy + e[:, 6] * dy * dy
                else:  # the pixel's ray (gx, gy, 1) meets the surfel's plane at (u, v)
                    gx, gy = (px - cx) / f, (py - cy) / f
                    k = [e[:, 4] - gx * e[:, 6], e[:, 7] - gx * e[:, 9], e[:, 10] - gx * e[:, 12]]
                    l = [e[:, 5] - gy * e[:, 6], e[:, 8] - gy * e[:, 9], e[:, 11] - gy * e[:, 12]]
                    n = k[0] * l[1] - k[1] * l[0]
                    u, v = (k[1] * l[2] - k[2] * l[1]) / n, (k[2] * l[0] - k[0] * l[2]) / n
                    r3, r2 = u * u + v * v, 2 * (dx * dx + dy * dy)
                    z = torch.where(r3 <= r2, e[:, 6] * u + e[:, 9] * v + e[:, 12], z)
                    rho = torch.minimum(torch.nan_to_num(r3, nan=1e300, posinf=1e300), r2)
                al = torch.where(rho <= e[:, 2], (o[i][:, None] * torch.exp(-0.5 * rho)).clamp_max(0.99), torch.zeros_like(rho))
                after = T * torch.cumprod(1 - al, 0)
                go = (after >= 1e-4) & ~done
                before = torch.cat([T[None], after[:-1]])
                wt = torch.where(go, al * before, torch.zeros_like(al))
                C += col[i].T @ wt
                Z += (wt * torch.where(wt > 0, z, torch.zeros_like(z))).sum(0)
                T = torch.where(go, after, torch.full_like(after, 2.0)).amin(0).minimum(T)
                done = ~go[-1]
                if bool(done.all()):
                    break
            shape = (y1 - y0, x1 - x0)
            for ch in range(3):
                rgb[ch, y0:y1, x0:x1] = (C[ch] + T * bg[ch]).view(shape)
            dep[y0:y1, x0:x1], tr[y0:y1, x0:x1] = Z.view(shape), T.view(shape)
    return rgb, dep, tr


def _net64(feat, tiles, params, h, w):
    """The network on each tile's 28 x 28 window in 64 bits: (n, 4, 16, 16) outputs, the tiles' inputs and the pixels inside the image."""
    t = tiles.to(torch.int64)
    f, y0, x0 = t >> 24, ((t >> 12) & 4095) * 16 - 6, (t & 4095) * 16 - 6
    a = torch.arange(28, device="cuda")
    ys, xs = (y0[:, None] + a)[:, :, None], (x0[:, None] + a)[:, None, :]
    ins = ((ys >= 0) & (ys < h) & (xs >= 0) & (xs < w)).double()[:, None]
    win = feat[f[:, None, None], ys.clamp(0, h - 1), xs.clamp(0, w - 1)][..., :6].double().permute(0, 3, 1, 2) * ins
    v, at = win, 0
    for l, (ci, co) in enumerate(((6, 32), (32, 32), (32, 32), (32, 32), (32, 32), (32, 4))):
        wt = params[at:at + co * 9 * ci].view(co, 3, 3, ci).permute(0, 3, 1, 2)
        b = params[at + co * 9 * ci:at + co * 9 * ci + co]
        at += co * 9 * ci + co
        e = 28 - 2 * l
        cols = torch.nn.functional.unfold(v, 3)  # (n, ci * 9, (e - 2)^2)
        v = (wt.reshape(co, ci * 9) @ cols + b[:, None]).view(-1, co, e - 2, e - 2)
        if l < 5:
            v = v.relu() * ins[:, :, l + 1:27 - l, l + 1:27 - l]
    return v, win[:, :, 6:22, 6:22], ins[:, :, 6:22, 6:22]


def exact(case, seed):
    g, call = _gen(seed), case["call"]
    if call in ("stereo", "mono", "two_pass"):
        w, h, f = case["w"], case["h"], case["f"]
        if w * h > 2.1e6 or case["n"] > 1600000:
            return None  # too many pixels for a few seconds
        sc = _scene(g, case["scene"], case["n"], case["sh"], case.get("ellipsoids", False))
        dom, aff = _head(seed, case["scene"], case.get("toe", 0.0))
        bg = (0.2, 0.3, 0.4) if call == "mono" else (0.0, 0.0, 0.0)
        rgb, dep, tr = _exact_view(sc, dom, w, h, f, bg)
        if call == "mono":
            return {"rgb": rgb, "depth": dep, "trans": tr}
        # a stereo frame's other eye copies pixels to where 32-bit arithmetic rounds them: no 64-bit value
        other = _exact_view(sc, aff, w, h, f)[0] if call == "two_pass" else None
        out = {"rgb_dom": rgb, "depth_dom": dep, "trans_dom": tr, "rgb_aff": other}
        if call == "stereo":
            out.update(cls_aff=None, roi_rects=None, roi_count=None, edge_widths=None)
        return out
    if call == "batch":
        return None  # as stereo, several times over
    h, w = case["h"], case["w"]
    if call == "infer":
        feat = _features(g, case["frames"], h, w)
        tiles = _tiles(g, feat, case["tiles"])
        params = torch.from_numpy(_weights(g)).cuda().double()
        out, win, ins = [], [], []
        for part in tiles.split(512):
            for keep, v in zip((out, win, ins), _net64(feat, part, params, h, w)):
                keep.append(v)
        out, win, ins = torch.cat(out), torch.cat(win), torch.cat(ins)
        fill = torch.zeros(case["frames"], 3, h, w, dtype=torch.float64, device="cuda")
        t = tiles.to(torch.int64)
        a = torch.arange(16, device="cuda")
        ys, xs = (((t >> 12) & 4095) * 16)[:, None, None] + a[:, None], ((t & 4095) * 16)[:, None, None] + a
        ys, xs = ys.expand(-1, 16, 16), xs.expand(-1, 16, 16)
        fr = (t >> 24)[:, None, None].expand(-1, 16, 16)
        m = ins[:, 0] > 0
        fill.permute(0, 2, 3, 1)[fr[m], ys[m], xs[m]] = (win[:, :3] + out[:, :3]).permute(0, 2, 3, 1)[m]
        return {"fill": fill, "gate": (out[:, 3:] * ins).sum((1, 2, 3)) / ins.sum((1, 2, 3))}
    if call == "train":
        feat, target, plain, tiles, w0, m0, v0 = _train_inputs(case, g)
        params = torch.from_numpy(w0).cuda().double().requires_grad_()
        out, win, ins = _net64(feat, tiles, params, h, w)
        t = tiles.to(torch.int64)
        a = torch.arange(16, device="cuda")
        ys = ((((t >> 12) & 4095) * 16)[:, None, None] + a[:, None]).clamp_max(h - 1)
        xs = (((t & 4095) * 16)[:, None, None] + a).clamp_max(w - 1)
        pick = lambda img: img.permute(0, 2, 3, 1)[(t >> 24)[:, None, None], ys, xs].double().permute(0, 3, 1, 2)
        tg, pl = pick(target), pick(plain)
        hole = (win[:, 4:5] > 0.5).double() * ins
        fill, n = win[:, :3] + out[:, :3], tiles.numel()
        holes = hole.sum((1, 2, 3))
        with torch.no_grad():
            mse = [((v - tg) ** 2 * hole).sum((1, 2, 3)) / (3 * holes).clamp_min(1) for v in (fill.clamp_min(0), pl)]
            mse[0] = torch.where(holes > 0, mse[0], torch.ones_like(holes))
            psnr = [torch.where(v > 0, -10 * torch.log10(v.clamp_min(1e-300)), torch.full_like(v, 1e9)) for v in mse]
            label = ((psnr[0] >= psnr[1] - 0.5) & (psnr[0] >= 30)).double()
        l1 = ((fill - tg).abs() * hole).sum() / (3 * hole.sum().clamp_min(1))
        gate = (out[:, 3:] * ins).sum((1, 2, 3)) / ins.sum((1, 2, 3))
        bce = torch.nn.functional.binary_cross_entropy_with_logits(gate, label)
        loss = l1 + ADAM["gate_weight"] * bce
        grad, = torch.autograd.grad(loss, params)
        m = ADAM["beta1"] * torch.from_numpy(m0).cuda().double() + (1 - ADAM["beta1"]) * grad
        v = ADAM["beta2"] * torch.from_numpy(v0).cuda().double() + (1 - ADAM["beta2"]) * grad ** 2
        k = STEPS + 1
        step = (m / (1 - ADAM["beta1"] ** k)) / ((v / (1 - ADAM["beta2"] ** k)).sqrt() + ADAM["eps"])
        p = params.detach()
        return {"loss": torch.stack([loss, l1, bce, label.mean()]).detach().cpu().numpy(), "gradients": grad.cpu().numpy(),
                "weights": (p - ADAM["lr"] * (step + ADAM["weight_decay"] * p)).cpu().numpy()}
    if call == "ssim":
        a, b = (t.double()[:, None] for t in _ssim_inputs(case, g))
        x = torch.arange(-5, 6, dtype=torch.float64, device="cuda")
        k = torch.exp(-x * x / 4.5)
        k = k / k.sum()

        def blur(t):  # separable 11-tap window, zero padding
            t = sum(k[i] * torch.nn.functional.pad(t, (5, 5, 0, 0))[..., i:i + t.shape[-1]] for i in range(11))
            return sum(k[i] * torch.nn.functional.pad(t, (0, 0, 5, 5))[..., i:i + t.shape[-2], :] for i in range(11))
        ma, mb = blur(a), blur(b)
        va, vb, cov = blur(a * a) - ma * ma, blur(b * b) - mb * mb, blur(a * b) - ma * mb
        c1, c2 = 1e-4, 9e-4
        return ((2 * ma * mb + c1) * (2 * cov + c2) / ((ma * ma + mb * mb + c1) * (va + vb + c2))).mean()
    # the warp: every pixel's landing place and depth, the nearest one wins
    rgb, dep, tr = (t.double() for t in _warp_inputs(case, g))
    dom, aff = _head(seed, "object")
    f, cx, cy = case["f"], (w - 1) / 2, (h - 1) / 2
    cov = 1 - tr
    solid = cov >= 0.5
    z = torch.where(solid, dep / cov.clamp_min(0.5), torch.ones_like(dep))
    y, x = torch.meshgrid(torch.arange(h, dtype=torch.float64, device="cuda"), torch.arange(w, dtype=torch.float64, device="cuda"), indexing="ij")
    p = torch.stack([(x - cx) / f * z, (y - cy) / f * z, z], -1)
    rel = torch.tensor(aff.R.T @ dom.R, device="cuda")
    off = torch.tensor(aff.R.T @ (dom.t - aff.t), device="cuda")
    q = p @ rel.T + solid[..., None] * off
    u = torch.floor(f * q[..., 0] / q[..., 2] + cx + 0.5).long()
    v = torch.floor(f * q[..., 1] / q[..., 2] + cy + 0.5).long()
    ok = (q[..., 2] > torch.where(solid, 0.2, 0.0)) & (u >= 0) & (u < w) & (v >= 0) & (v < h)
    zq = torch.where(solid, q[..., 2], torch.full_like(z, math.inf)).flatten()
    order = torch.argsort(zq, stable=True)
    order = order[ok.flatten()[order]]
    rank = torch.full((h * w,), h * w, dtype=torch.int64, device="cuda")
    rank.scatter_reduce_(0, (v * w + u).flatten()[order], torch.arange(order.numel(), device="cuda"), "amin")
    hit = rank < h * w
    src = order[rank.clamp_max(order.numel() - 1)]
    out = torch.where(hit, rgb.view(3, -1)[:, src], torch.zeros(3, 1, dtype=torch.float64, device="cuda"))
    depth = torch.where(hit, zq[src], torch.zeros_like(zq))
    return {"rgb": out.view(3, h, w), "depth": depth.view(h, w), "hole": None}
