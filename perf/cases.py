"""The work that users of this framework have it do, as measured cases.

Every case goes through the public front ends (Renderer, render, Tracker,
MappingLoss, Decoder, DistillLoss, Adam, VoxelMap, ICP, AnchorStats,
AnchorUpdate, Spawner) on the seeded scenes of paper_2505_18992_gb300.scenes.

  listed()             the cases
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  inputs and handles a program holds before the call
  run(state)           one pass; its outputs
  work(case)           bytes and flops the pass cannot do without
  exact(case, seed)    the outputs in 64 bits from plain torch, where that is quick
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2505_18992_gb300 import scenes
from paper_2505_18992_gb300.anchors import AnchorStats, AnchorUpdate, Spawner
from paper_2505_18992_gb300.decode import Decoder
from paper_2505_18992_gb300.fusion import Adam, DistillLoss
from paper_2505_18992_gb300.icp import ICP, VoxelMap
from paper_2505_18992_gb300.loss import MappingLoss
from paper_2505_18992_gb300.render import Intrinsics, Renderer, render
from paper_2505_18992_gb300.tracking import Tracker

DEV = "cuda"
F64 = torch.float64
NAMES = ("means", "scales", "quats", "opacities", "colors")


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------

def listed():
    return [
        # a preview of a handful of Gaussians in three ragged views: the smallest call,
        # all latency and launches
        {"name": "view_tiny", "kind": "view", "scene": "random", "n": 300, "width": 97, "height": 61, "views": 3},
        # one training step on a small scene through autograd: 10,000 Gaussians at 320x240
        {"name": "render_small", "kind": "render", "scene": "planes", "n": 10_000, "width": 320, "height": 240,
         "views": 1},
        # coarse tracking of a small frame: ten pose iterations replayed from one CUDA graph
        {"name": "track_small", "kind": "track", "scene": "planes", "n": 10_000, "width": 320, "height": 240,
         "iters": 10},
        # coarse tracking against the indoor room, the frame size of the room sequences
        {"name": "track_room", "kind": "track", "scene": "room", "n": 1_000_000, "width": 1200, "height": 680,
         "iters": 10},
        # a mapping step on the room: render, the full loss, the backward to every Gaussian parameter
        {"name": "map_room", "kind": "map", "scene": "room", "n": 1_000_000, "width": 1200, "height": 680},
        # a forward-only render (spawning masks, previews) at the ragged KITTI frame size
        {"name": "view_street", "kind": "view", "scene": "street", "n": 400_000, "width": 1241, "height": 376,
         "views": 1},
        # eight keyframes of a 2M-Gaussian submap trained in one call through autograd
        {"name": "render_keyframes", "kind": "render", "scene": "keyframes", "n": 2_000_000, "width": 640,
         "height": 480, "views": 8},
        # anchor decode and its backward on the tensor cores: a street submap
        {"name": "decode_bf16", "kind": "decode", "anchors": 100_000, "k": 10, "bf16": True, "half": False},
        # the same in FP32 on an odd, smaller number of anchors
        {"name": "decode_fp32", "kind": "decode", "anchors": 37_511, "k": 10, "bf16": False, "half": False},
        # one step of submap fusion: two 50,000-anchor submaps decoded, rendered into four full-HD
        # keyframes, distilled, back-propagated and stepped
        {"name": "fusion_pair", "kind": "fusion", "anchors": 50_000, "width": 1920, "height": 1080, "views": 4},
        # fine tracking: the map's voxel hash rebuilt and a 64-beam sweep registered against it
        {"name": "icp_street", "kind": "icp", "map": 1_000_000, "beams": 64, "azimuths": 1800, "iters": 50},
        # anchor maintenance after a keyframe: statistics, pruning and growth, spawning
        {"name": "anchors_street", "kind": "anchors", "anchors": 100_000, "width": 1200, "height": 680,
         "gauss": 300_000, "samples": 50_000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _frame(rng, lo_px, hi_px):
    """An image size, any parity, of lo_px..hi_px pixels and aspect 1..3."""
    px, aspect = math.exp(rng.uniform(math.log(lo_px), math.log(hi_px))), rng.uniform(1.0, 3.0)
    w = max(16, int(round(math.sqrt(px * aspect))))
    return w, max(16, int(px / w))


def draw(rng):
    kind = rng.choice(("view", "render", "render", "track", "map", "decode", "decode", "fusion", "icp", "anchors"))
    if kind in ("view", "render"):
        scene = rng.choice(("random", "planes", "room", "street", "keyframes"))
        views = rng.randint(1, 4) if scene == "random" else rng.randint(2, 8) if scene == "keyframes" else 1
        w, h = _frame(rng, 5_000, 100_000 if scene in ("random", "planes") else 900_000 // views)
        n = _log(rng, 300, 20_000) if scene in ("random", "planes") else _log(rng, 20_000, 1_500_000)
        return {"kind": kind, "scene": scene, "n": n, "width": w, "height": h, "views": views}
    if kind in ("track", "map"):
        scene = rng.choice(("planes", "room", "street"))
        w, h = _frame(rng, 20_000, 100_000 if scene == "planes" else 800_000)
        n = _log(rng, 2_000, 20_000) if scene == "planes" else _log(rng, 50_000, 1_000_000)
        c = {"kind": kind, "scene": scene, "n": n, "width": w, "height": h}
        return {**c, "iters": rng.randint(3, 10)} if kind == "track" else c
    if kind == "decode":
        return {"kind": kind, "anchors": _log(rng, 50, 100_000), "k": rng.choice((10, 10, 5, 3)),
                "bf16": rng.random() < 0.6, "half": rng.random() < 0.3}
    if kind == "fusion":
        w, h = _frame(rng, 50_000, 2_000_000)
        return {"kind": kind, "anchors": _log(rng, 3_000, 50_000), "width": w, "height": h,
                "views": rng.randint(1, 4)}
    if kind == "icp":
        return {"kind": kind, "map": _log(rng, 30_000, 1_000_000), "beams": rng.choice((16, 32, 64)),
                "azimuths": rng.randint(300, 1800), "iters": rng.randint(10, 50)}
    w, h = _frame(rng, 40_000, 800_000)
    return {"kind": kind, "anchors": _log(rng, 2_000, 100_000), "width": w, "height": h,
            "gauss": _log(rng, 5_000, 300_000), "samples": _log(rng, 500, 50_000)}


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _dev(a, dtype=torch.float32):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype).to(DEV)


def _scene(c, seed):
    """The Gaussians and the camera(s) of a render-like case (numpy)."""
    n, w, h = c["n"], c["width"], c["height"]
    if c["scene"] == "random":
        return scenes.random_gaussians(n, w, h, 1.1 * w, seed, n_views=c["views"])
    if c["scene"] == "planes":
        return scenes.tiny_planes(n, w, h, 0.94 * w, seed)
    if c["scene"] == "room":
        return scenes.indoor_room(n, w, h, 0.5 * w, seed)
    if c["scene"] == "keyframes":
        return scenes.batched_keyframes(n, c["views"], w, h, 0.82 * w, seed=seed)
    # street: ground and facades in front of a car's camera
    rng = np.random.default_rng(seed)
    means = scenes.corridor_points(rng, n).astype(np.float32)[rng.permutation(n)]
    o = scenes.random_gaussians(n, w, h, 0.58 * w, seed)  # attributes of n Gaussians
    T = scenes.look_at([4.0, 0.0, 1.7], [5.0, 0.0, 1.7], [0, 0, 1])
    cam = scenes.Camera(w, h, 0.58 * w, 0.58 * w, w / 2.0, h / 2.0, T[None])
    return scenes.GaussianScene("street", means, o.scales, o.quats, o.opacities, o.colors, cam)


def _renderer(cam, g, T):
    r = Renderer(Intrinsics(cam.width, cam.height, cam.fx, cam.fy, cam.cx, cam.cy), n_views=T.shape[0], device=DEV)
    r.forward(*g, T, check=True)  # sizes the workspace once, as a program does
    return r


def _flat_mlp(mlp):
    return np.concatenate([np.asarray(p, np.float32).reshape(-1) for m in ("opacity", "color", "cov") for p in mlp[m]])


def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _upstream(seed, V, H, W):
    """Upstream gradients of the images: the scale of a mean loss, random signs and sizes."""
    gen, s = _generator(seed), 1.0 / (V * H * W)
    return [torch.randn(shape, generator=gen, device=DEV) * s for shape in ((V, 3, H, W), (V, H, W), (V, H, W))]


def _prepare_view(c, seed):
    sc = _scene(c, seed)
    g, T = [_dev(a) for a in sc.arrays()], _dev(sc.camera.T_cw, F64)
    r = _renderer(sc.camera, g, T)
    return {"r": r, "g": g, "T": T, "out": r.alloc_images()}


def _run_view(s):
    return s["r"].forward(*s["g"], s["T"], out=s["out"], check=False)


def _prepare_render(c, seed):
    sc = _scene(c, seed)
    g, T = [_dev(a) for a in sc.arrays()], _dev(sc.camera.T_cw, F64)
    r = _renderer(sc.camera, g, T)
    return {"r": r, "g": [t.requires_grad_(True) for t in g], "T": T,
            "up": _upstream(seed + 1, r.V, c["height"], c["width"])}


def _run_render(s):
    out = render(*s["g"], s["T"], s["r"])
    grads = torch.autograd.grad(out, s["g"], s["up"])
    return {"rgb": out[0].detach(), "depth": out[1].detach(), "alpha": out[2].detach(),
            "grads": dict(zip(NAMES, grads))}


def _moved(T, seed):
    """The pose 2 cm and 1 degree off, where tracking starts (or a target was taken)."""
    return scenes.perturb_pose(T[0], np.random.default_rng(seed + 100), 0.02, 1.0)[None]


def _prepare_track(c, seed):
    sc = _scene(c, seed)
    g, T, T0 = [_dev(a) for a in sc.arrays()], _dev(sc.camera.T_cw, F64), _dev(_moved(sc.camera.T_cw, seed), F64)
    r = _renderer(sc.camera, g, T)
    frame = r.forward(*g, T, check=True)
    tr = Tracker(r, g, T0.clone(), frame["rgb"].clone(), frame["depth"].clone())
    tr.prepare()
    tr.capture(c["iters"])
    return {"tr": tr, "T0": T0}


def _run_track(s):
    tr = s["tr"]
    tr.reset(s["T0"])
    tr.replay()
    return {"T": tr.T, "loss": tr.loss, "rgb": tr.out["rgb"], "depth": tr.out["depth"]}


def _prepare_map(c, seed):
    sc = _scene(c, seed)
    g, T = [_dev(a) for a in sc.arrays()], _dev(sc.camera.T_cw, F64)
    r = _renderer(sc.camera, g, T)
    frame = r.forward(*g, _dev(_moved(sc.camera.T_cw, seed), F64), check=True)
    out = r.alloc_images()
    return {"r": r, "g": g, "T": T, "out": out, "loss": MappingLoss(1, c["width"], c["height"], device=DEV),
            "rgb": frame["rgb"].clone(), "depth": frame["depth"].clone(),
            "d_rgb": torch.empty_like(out["rgb"]), "d_depth": torch.empty_like(out["depth"]),
            "grads": {k: torch.zeros_like(t) for k, t in zip(NAMES, g)}}


def _run_map(s):
    r, g, out, grads = s["r"], s["g"], s["out"], s["grads"]
    for t in grads.values():
        t.zero_()
    r.forward(*g, s["T"], out=out, check=False)
    loss = s["loss"](out["rgb"], s["rgb"], out["depth"], s["depth"], g[1], d_rgb=s["d_rgb"], d_depth=s["d_depth"],
                     d_scales=grads["scales"])
    r.backward(*g, s["T"], out, s["d_rgb"], s["d_depth"], None, grads=grads)
    return {"loss": loss, "rgb": out["rgb"], "depth": out["depth"], "alpha": out["alpha"], "grads": grads}


def _street_anchors(c, seed):
    return scenes.street_anchors(c["anchors"], seed=seed, k=c["k"])


def _decode_upstream(c, seed, n_anchors):
    """The upstream gradients of a decode case."""
    gen, cap = _generator(seed + 1), max(n_anchors * c["k"], 1)
    shapes = {"means": (cap, 3), "scales": (cap, 3), "quats": (cap, 4), "opacities": (cap,), "colors": (cap, 3)}
    return {k: torch.randn(shapes[k], generator=gen, device=DEV) for k in NAMES}


def _prepare_decode(c, seed):
    sc = _street_anchors(c, seed)
    feats = _dev(sc.features, torch.bfloat16 if c["half"] else torch.float32)
    inp = (_dev(sc.anchors), feats, _dev(sc.scaling), _dev(sc.offsets), _dev(_flat_mlp(sc.mlp)))
    d = Decoder(c["k"], bf16=c["bf16"], device=DEV)
    out = d.alloc_outputs(sc.n)
    for t in out.values():
        t.zero_()  # rows past the decoded count stay as they are
    up = _decode_upstream(c, seed, sc.n)
    res = {"features": torch.zeros(feats.shape, device=DEV), "offsets": torch.zeros_like(inp[3]),
           "scaling": torch.zeros_like(inp[2]), "params": torch.zeros_like(inp[4])}
    return {"d": d, "inp": inp, "cam": sc.camera, "T": _dev(sc.camera.T_cw[0], F64), "out": out, "up": up, "res": res}


def _run_decode(s):
    out = s["d"].forward(*s["inp"], s["cam"], s["T"], out=s["out"], sync=False)
    for t in s["res"].values():
        t.zero_()
    res = s["d"].backward(*s["inp"], s["cam"], s["T"], out, s["up"], res=s["res"])
    return {"out": {k: out[k] for k in (*NAMES, "n_dev", "src_index")}, "grads": res}


def _prepare_fusion(c, seed):
    # two submaps of a street that overlap by 10 m, and keyframes in the overlap facing a facade
    m, w, h = c["views"], c["width"], c["height"]
    T = _dev(np.stack([scenes.look_at([57.0 + 2.0 * i, 0.0, 1.7], [57.0 + 2.0 * i, 10.0, 1.7], [0, 0, 1])
                       for i in range(m)]), F64)
    subs, r = [], None
    for j, (x0, x1) in enumerate(((0.0, 62.5), (52.5, 125.0))):
        sc = scenes.street_anchors(c["anchors"], w, h, 0.52 * w, length=x1 - x0, x0=x0, seed=2 * seed + j,
                                   mlp_seed=seed)
        sc.camera.T_cw = T[:1].cpu().numpy()
        inp = (_dev(sc.anchors), _dev(sc.features), _dev(sc.scaling), _dev(sc.offsets), _dev(_flat_mlp(sc.mlp)))
        d = Decoder(sc.k, bf16=True, device=DEV)
        out = d.forward(*inp, sc.camera, T[0], sync=False)
        if r is None:
            r = Renderer(Intrinsics(w, h, 0.52 * w, 0.52 * w, w / 2.0, h / 2.0), n_views=m, device=DEV)
        img = r.alloc_images()
        r.forward(*(out[k] for k in NAMES), T, n_dev=out["n_dev"], out=img, check=True)
        res = {"features": torch.zeros_like(inp[1]), "offsets": torch.zeros_like(inp[3]),
               "scaling": torch.zeros_like(inp[2]), "params": torch.zeros_like(inp[4])}
        subs.append({"d": d, "inp": inp, "cam": sc.camera, "out": out, "img": img, "res": res,
                     "opts": [Adam(inp[1], res["features"], lr=1e-4), Adam(inp[4], res["params"], lr=1e-5)],
                     "grads": {k: torch.zeros_like(out[k]) for k in NAMES},
                     "d_rgb": torch.empty_like(img["rgb"]), "d_depth": torch.empty_like(img["depth"])})
    return {"r": r, "T": T, "subs": subs, "dist": DistillLoss(m, w, h, device=DEV)}


def _run_fusion(s):
    r, T, (a, b) = s["r"], s["T"], s["subs"]
    for u in s["subs"]:
        o = u["d"].forward(*u["inp"], u["cam"], T[0], out=u["out"], sync=False)
        r.forward(*(o[k] for k in NAMES), T, n_dev=o["n_dev"], out=u["img"], check=False)
    loss = s["dist"](a["img"]["rgb"], b["img"]["rgb"], a["img"]["depth"], b["img"]["depth"], a["d_rgb"], b["d_rgb"],
                     a["d_depth"], b["d_depth"])
    for u in s["subs"]:
        o = u["out"]
        for t in u["grads"].values():
            t.zero_()
        r.backward(*(o[k] for k in NAMES), T, u["img"], u["d_rgb"], u["d_depth"], None, grads=u["grads"],
                   n_dev=o["n_dev"])
        u["d"].backward(*u["inp"], u["cam"], T[0], o, u["grads"], res=u["res"])
        for opt in u["opts"]:
            opt.step()
    return {"loss": loss, "subs": [{"rgb": u["img"]["rgb"], "depth": u["img"]["depth"], "features": u["inp"][1],
                                    "params": u["inp"][4]} for u in s["subs"]]}


def _prepare_icp(c, seed):
    sc = scenes.street_lidar(c["map"], c["beams"], c["azimuths"], seed=seed)
    T0 = _dev(sc.T_init, F64)
    return {"map": VoxelMap(_dev(sc.map_points), 1.0), "scan": _dev(sc.scan), "T0": T0, "T": T0.clone(),
            "icp": ICP(len(sc.scan), 0.5, 1.5, 1.0, 0.3, iterations=c["iters"], eps=1e-4, device=DEV)}


def _run_icp(s):
    s["map"].rebuild()  # the map's Gaussians moved since the last frame
    s["T"].copy_(s["T0"])
    return s["icp"].register(s["map"], s["scan"], s["T"])


def _anchor_step(c, seed):
    return scenes.anchor_step(c["anchors"], seed=seed)


def _prepare_anchors(c, seed):
    st = _anchor_step(c, seed)
    fr = scenes.keyframe_spawn(c["width"], c["height"], 0.5 * c["width"], c["gauss"], seed + 1)
    up = AnchorUpdate(len(st.anchors), len(st.src_index), 2.5e-3, 0.3, 0.2, device=DEV)
    sp = Spawner(fr.width, fr.height, fr.fx, fr.fy, fr.cx, fr.cy, 0.5, 0.1, 0.05, 0.04, c["samples"], device=DEV)
    for t in (up.keep, up.grown, sp.anchors):
        t.zero_()  # rows past the counts stay as they are
    return {"k": st.k, "src": _dev(st.src_index, torch.int32), "grads": _dev(st.grads), "opac": _dev(st.opacities),
            "vis": _dev(st.visible, torch.int32), "means": _dev(st.means), "stats": AnchorStats(len(st.anchors), DEV),
            "amap": VoxelMap(_dev(st.anchors), 0.2), "gmap": VoxelMap(_dev(fr.gauss_means), 0.05), "up": up, "sp": sp,
            "frame": (_dev(fr.alpha), _dev(fr.depth), _dev(fr.depth_in), _dev(fr.T_cw, F64))}


def _run_anchors(s):
    s["stats"].reset()
    s["stats"].accumulate(s["k"], s["src"], s["grads"], s["opac"], s["vis"])
    keep, grown, counts = s["up"](s["stats"], s["k"], s["src"], s["means"], s["amap"])
    new, _, n_new = s["sp"](*s["frame"], s["gmap"])
    return {"stats": s["stats"].arrays(), "keep": keep, "grown": grown, "counts": counts, "new": new, "n_new": n_new[:1]}


_KINDS = {"view": (_prepare_view, _run_view), "render": (_prepare_render, _run_render),
          "track": (_prepare_track, _run_track), "map": (_prepare_map, _run_map),
          "decode": (_prepare_decode, _run_decode), "fusion": (_prepare_fusion, _run_fusion),
          "icp": (_prepare_icp, _run_icp), "anchors": (_prepare_anchors, _run_anchors)}


def prepare(case, seed):
    make, go = _KINDS[case["kind"]]
    return {"run": go, **make(case, int(seed))}


def run(state):
    return state["run"](state)


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------

# (share of the Gaussians in view, mean footprint in pixels over (focal length)^2) per scene: the
# generators' means, for estimates of the pixel-Gaussian pairs that blend
_SEEN = {"random": (0.9, 5.0e-4), "planes": (0.6, 1.2e-3), "room": (0.17, 1.3e-3), "street": (0.4, 1.0e-4),
         "keyframes": (0.15, 1.5e-3)}


def _pairs(scene, n, w, h, views, f):
    """Estimated blended pixel-Gaussian pairs: coverage, up to where a pixel's transmittance runs out."""
    share, area = _SEEN[scene]
    px = w * h
    return views * px * min(70.0, share * n * (area * f * f + 3.0) / px)


def _render_work(scene, n, w, h, views, f, backward):
    """Gaussians in, images out; backward: upstream images in, gradients out.  11 flops per blended
    pair forward and 40 backward, on top of 17 for the pair's opacity in each."""
    px, pairs = views * w * h, _pairs(scene, n, w, h, views, f)
    if not backward:
        return {"bytes": 56 * n + 32 * px, "flops": 28 * pairs}
    return {"bytes": 112 * n + 52 * px, "flops": 85 * pairs}


def work(case):
    c, kind = case, case["kind"]
    if kind in ("view", "render", "track", "map"):
        f = {"random": 1.1, "planes": 0.94, "room": 0.5, "keyframes": 0.82, "street": 0.58}[c["scene"]] * c["width"]
        w = _render_work(c["scene"], c["n"], c["width"], c["height"], c.get("views", 1), f, kind != "view")
        if kind == "track":  # the frame once; per iteration the pairs, no gradient leaves but the pose's
            px = c["width"] * c["height"]
            return {"bytes": 56 * c["n"] + 32 * px, "flops": c["iters"] * w["flops"]}
        if kind == "map":  # the target in; two separable 11-tap blurs of 8 fields per colour pixel
            px = c["width"] * c["height"]
            return {"bytes": w["bytes"] + 16 * px, "flops": w["flops"] + 3 * px * 8 * 44}
        return w
    if kind == "decode":
        A, k = c["anchors"], c["k"]
        feat = 64 if c["half"] else 128
        macs = 3 * 36 * 32 + 32 * 11 * k
        seen = 0.55 * A  # anchors in view; about half of their Gaussians are valid
        gauss = 0.5 * k * seen
        return {"bytes": A * (12 + feat + 12 + 12 * k) + gauss * (60 + 56) + A * (128 + 12 + 12 * k),
                "flops": 6 * macs * seen}
    if kind == "fusion":
        A, px = c["anchors"], c["views"] * c["width"] * c["height"]
        pairs = 2 * _pairs("street", 2 * A, c["width"], c["height"], c["views"], 0.52 * c["width"])
        return {"bytes": 2 * (A * (12 + 128 + 12 + 120) + 32 * px + A * 128 * 2), "flops": 85 * pairs +
                2 * 6 * 0.3 * A * (3 * 36 * 32 + 320 * 11)}
    if kind == "icp":
        scan = c["beams"] * c["azimuths"]
        return {"bytes": 12 * c["map"] + 16 * c["map"] + 12 * scan, "flops": c["iters"] * 1300 * 30 * 8}
    n = 5 * c["anchors"]
    return {"bytes": 24 * n + 16 * c["anchors"] + 12 * n + 12 * c["width"] * c["height"] + 24 * c["samples"],
            "flops": 10 * n}


# --------------------------------------------------------------------------
# the same outputs in 64 bits
# --------------------------------------------------------------------------

def _exact_images(c, seed, backward):
    """Dense splatting of a small scene in 64 bits: every pixel against every Gaussian in depth
    order (the rules and default options of the renderer's header), a few image rows at a time."""
    sc = _scene(c, seed)
    cam, (H, W) = sc.camera, (c["height"], c["width"])
    if sc.n * cam.pixels > 2_000_000_000:
        return None
    leaves = [_dev(a, F64).requires_grad_(backward) for a in sc.arrays()]
    means, scales, quats, opac, colors = leaves
    up = [t.to(F64) for t in _upstream(seed + 1, cam.n_views, H, W)] if backward else None
    images = {"rgb": torch.empty((cam.n_views, 3, H, W), dtype=F64, device=DEV)}
    images.update({k: torch.empty((cam.n_views, H, W), dtype=F64, device=DEV) for k in ("depth", "alpha", "t_final")})
    grads = [torch.zeros_like(t) for t in leaves]
    rows = max(1, int(12_000_000 // (W * sc.n)))
    for v in range(cam.n_views):
        T = _dev(cam.T_cw[v], F64)
        R = T[:3, :3]
        for y0 in range(0, H, rows):
            y1 = min(H, y0 + rows)
            p = means @ R.T + T[:3, 3]
            order = torch.argsort(p[:, 2].detach().float(), stable=True)
            order = order[p[order, 2].detach() > 0.2]
            x, y, z = p[order].unbind(1)
            q = quats[order] / quats[order].norm(dim=1, keepdim=True)
            a, b, e, d = q.unbind(1)
            Rq = torch.stack([1 - 2 * (e * e + d * d), 2 * (b * e - a * d), 2 * (b * d + a * e),
                              2 * (b * e + a * d), 1 - 2 * (b * b + d * d), 2 * (e * d - a * b),
                              2 * (b * d - a * e), 2 * (e * d + a * b), 1 - 2 * (b * b + e * e)], 1).reshape(-1, 3, 3)
            zero = torch.zeros_like(z)
            J = torch.stack([cam.fx / z, zero, -cam.fx * x / z ** 2, zero, cam.fy / z, -cam.fy * y / z ** 2],
                            1).reshape(-1, 2, 3)
            K = J @ R @ Rq * scales[order][:, None, :]
            S = K @ K.transpose(1, 2) + 0.3 * torch.eye(2, dtype=F64, device=DEV)
            det = S[:, 0, 0] * S[:, 1, 1] - S[:, 0, 1] ** 2
            jj, ii = torch.meshgrid(torch.arange(y0, y1, device=DEV), torch.arange(W, device=DEV), indexing="ij")
            dx = ii.reshape(-1, 1) + 0.5 - (cam.fx * x / z + cam.cx)
            dy = jj.reshape(-1, 1) + 0.5 - (cam.fy * y / z + cam.cy)
            power = (S[:, 1, 1] * dx * dx - 2 * S[:, 0, 1] * dx * dy + S[:, 0, 0] * dy * dy) / det
            al = torch.clamp(opac[order] * torch.exp(-0.5 * power), max=0.99)
            al = torch.where(al.detach() < 1.0 / 255.0, torch.zeros_like(al), al)
            after = torch.cumprod(1 - al, 1)
            keep = (torch.cumsum((after.detach() < 1e-4) & (al.detach() > 0), 1) == 0).to(F64)
            al = al * keep
            after = torch.cumprod(1 - al, 1)
            before = torch.cat([torch.ones_like(after[:, :1]), after[:, :-1]], 1)
            wgt = al * before
            t_fin = after[:, -1]
            part = {"rgb": (wgt @ colors[order]).T.reshape(3, y1 - y0, W), "depth": (wgt @ z).reshape(y1 - y0, W),
                    "alpha": (1 - t_fin).reshape(y1 - y0, W), "t_final": t_fin.reshape(y1 - y0, W)}
            images["rgb"][v, :, y0:y1] = part["rgb"].detach()
            for k in ("depth", "alpha", "t_final"):
                images[k][v, y0:y1] = part[k].detach()
            if backward:
                L = (part["rgb"] * up[0][v, :, y0:y1]).sum() + (part["depth"] * up[1][v, y0:y1]).sum() + \
                    (part["alpha"] * up[2][v, y0:y1]).sum()
                for t, g in zip(grads, torch.autograd.grad(L, leaves, allow_unused=True)):
                    if g is not None:
                        t += g
    if not backward:
        return {**images, "n_contrib": None, "n_iter": None}
    return {"rgb": images["rgb"], "depth": images["depth"], "alpha": images["alpha"],
            "grads": dict(zip(NAMES, grads))}


def _exact_decode(c, seed):
    """The decoder's MLPs, heads and their gradients in 64 bits (its bfloat16 form rounds the network's
    input, weights and hidden values; gradients pass through the rounding)."""
    sc, k = _street_anchors(c, seed), c["k"]
    cam = sc.camera

    def rnd(t):
        return t + (t.detach().to(torch.bfloat16).to(F64) - t.detach()) if c["bf16"] else t

    feats = _dev(sc.features, torch.bfloat16 if c["half"] else torch.float32).to(F64).requires_grad_(True)
    scal, offs = _dev(sc.scaling, F64).requires_grad_(True), _dev(sc.offsets, F64).requires_grad_(True)
    params = _dev(_flat_mlp(sc.mlp), F64).requires_grad_(True)
    x, T = _dev(sc.anchors, F64), _dev(cam.T_cw[0], F64)
    p = x @ T[:3, :3].T + T[:3, 3]
    u, v = cam.fx * p[:, 0] / p[:, 2] + cam.cx, cam.fy * p[:, 1] / p[:, 2] + cam.cy
    gw, gh = 0.15 * cam.width, 0.15 * cam.height
    seen = torch.nonzero((p[:, 2] > 0.2) & (u >= -gw) & (u <= cam.width + gw) & (v >= -gh) & (v <= cam.height + gh))[:, 0]
    d = x[seen] + T[:3, :3].T @ T[:3, 3]
    delta = d.norm(dim=1, keepdim=True)
    inp, at, heads = rnd(torch.cat([feats[seen], d / delta, delta], 1)), 0, []
    for width in (k, 3 * k, 7 * k):
        w1, b1 = params[at:at + 1152].reshape(32, 36), params[at + 1152:at + 1184]
        at += 1184
        w2, b2 = params[at:at + 32 * width].reshape(width, 32), params[at + 32 * width:at + 33 * width]
        at += 33 * width
        heads.append(rnd(torch.relu(inp @ rnd(w1).T + b1)) @ rnd(w2).T + b2)
    op, col, cov = torch.tanh(heads[0]), torch.sigmoid(heads[1]).reshape(-1, k, 3), heads[2].reshape(-1, k, 7)
    l = scal[seen][:, None, :]
    got = {"means": x[seen][:, None, :] + offs[seen] * l, "scales": torch.sigmoid(cov[..., :3]) * l,
           "quats": cov[..., 3:] / cov[..., 3:].norm(dim=-1, keepdim=True), "opacities": op, "colors": col}
    valid = op.detach() > 0
    up = _decode_upstream(c, seed, sc.n)
    n, L, out = int(valid.sum()), torch.zeros((), dtype=F64, device=DEV), {}
    for key in NAMES:
        rows = got[key][valid]
        out[key] = torch.zeros(up[key].shape, dtype=F64, device=DEV)
        out[key][:n] = rows.detach()
        L = L + (rows * up[key][:n].to(F64)).sum()
    g = torch.autograd.grad(L, (feats, offs, scal, params))
    return {"out": {**out, "n_dev": None, "src_index": None},
            "grads": dict(zip(("features", "offsets", "scaling", "params"), g))}


def _exact_anchors(c, seed):
    """The statistics' sums in 64 bits; the rest of the case is decisions, indices and voxel centres."""
    st = _anchor_step(c, seed)
    a = _dev(st.src_index, torch.int64) // st.k
    norm = _dev(st.grads, F64).norm(dim=1) * (_dev(st.visible, F64) > 0)
    zero = torch.zeros(len(st.anchors), dtype=F64, device=DEV)
    return {"stats": {"g_sum": zero.index_add(0, a, norm), "o_sum": zero.index_add(0, a, _dev(st.opacities, F64)),
                      "g_cnt": None, "visits": None},
            "keep": None, "grown": None, "counts": None, "new": None, "n_new": None}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("view", "render"):
        return _exact_images(case, int(seed), kind == "render")
    if kind == "decode":
        return _exact_decode(case, int(seed))
    if kind == "anchors":
        return _exact_anchors(case, int(seed))
    return None  # a million Gaussians, or an iteration that feeds on its own results
