"""Workloads of the stitching library's public entry points, for timing and for comparing outputs.

``listed()`` holds the work that users of the library have it do: per-frame stitching from the
smallest rig to the largest, the options that are used with it (seam weights, FP16 bands, float
output, a cylindrical canvas), several rigs in one batch, host-resident video, the allocation-free
entry, the alignment loss with its gradient, and registration (features, matching, both chained).
``draw(rng)`` gives further cases of the same ranges.  Camera views are rendered on the GPU from one
random scene per seed, so that neighbouring views show the same content where they overlap.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_1810_03988_gb300 import LORB, Batch, Matcher, Rig, stitch


class Camera:
    def __init__(self, width, height, H, gain=1.0):
        self.width, self.height, self.H, self.gain = width, height, H, gain


def listed():
    stitch_u8 = {"kind": "stitch", "seam": False, "fp16": False, "float": False, "geo": 0}
    return [
        # a two-camera preview: the smallest rig in use, where launches and latency count
        {"name": "stitch_2x360p", **stitch_u8, "rig": "planar", "cams": 2, "w": 640, "h": 360, "f": 500.0,
         "step": 24.0, "cw": 1100, "ch": 400, "levels": 4},
        # the ordinary live panorama: four 1080p cameras
        {"name": "stitch_4x1080p", **stitch_u8, "rig": "planar", "cams": 4, "w": 1920, "h": 1080, "f": 1400.0,
         "step": 25.0, "cw": 5200, "ch": 1300, "levels": 5},
        # the largest rig: eight 4K cameras, 280 degrees
        {"name": "stitch_8x4k", **stitch_u8, "rig": "tangent", "cams": 8, "w": 3840, "h": 2160, "f": 4125.0,
         "step": 40.0, "cw": 24000, "ch": 2600, "levels": 6},
        # float output for further processing, seam masks, FP16 bands, odd sizes throughout
        {"name": "stitch_5x719_seam_fp16_float", "kind": "stitch", "rig": "tangent", "cams": 5, "w": 1277, "h": 719,
         "f": 1345.0, "step": 39.0, "cw": 4951, "ch": 863, "levels": 5, "seam": True, "fp16": True, "float": True,
         "geo": 3},
        # a wide-angle rig on the cylindrical canvas
        {"name": "stitch_cylinder_4x720p", **stitch_u8, "rig": "cylinder", "cams": 4, "w": 1280, "h": 720, "f": 900.0,
         "step": 30.0, "cw": 2528, "ch": 760, "levels": 5},
        # a server stitching eight independent rigs of uneven sizes per tick
        {"name": "batch_8_rigs", "kind": "batch", "rigs": 8, "geo": 0, "most": 2, "fp16": False, "float": False},
        # a caller that may not allocate device memory
        {"name": "static_2x360p", **stitch_u8, "kind": "static", "rig": "planar", "cams": 2, "w": 640, "h": 360,
         "f": 500.0, "step": 24.0, "cw": 1100, "ch": 400, "levels": 4},
        # host-resident video through pinned buffers, uploads and downloads overlapped
        {"name": "host_4x1080p", **stitch_u8, "kind": "host", "rig": "planar", "cams": 4, "w": 1920, "h": 1080,
         "f": 1400.0, "step": 25.0, "cw": 5200, "ch": 1300, "levels": 5},
        # one step of alignment refinement: overlap loss and its gradient
        {"name": "loss_4x1080p", "kind": "loss", "rig": "planar", "cams": 4, "w": 1920, "h": 1080, "f": 1400.0,
         "step": 25.0, "cw": 5200, "ch": 1300, "levels": 5, "geo": 0},
        # features of a whole 4K view
        {"name": "features_4k", "kind": "features", "w": 3840, "h": 2160, "points": 500, "areas": 1, "fast_t": 20},
        # matching and homography of two views with a thousand features each
        {"name": "match_1000", "kind": "match", "points": 1000, "tables": 8, "bits": 16, "iters": 1000},
        # registration of a small pair from its frames: features of both views, then the homography
        {"name": "register_2x360p", "kind": "register", "rig": "planar", "cams": 2, "w": 640, "h": 360, "f": 500.0,
         "step": 24.0, "cw": 1100, "ch": 400, "levels": 4, "geo": 0, "points": 300, "iters": 256},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_rig(rng, most_px, most_w=3840):
    """A rig of 2 to 8 cameras with overlapping neighbours whose canvas has at most most_px pixels."""
    while True:
        cams, w = rng.randint(2, 8), _log(rng, 320, most_w)
        h = int(w * rng.choice([9 / 16, 3 / 4, 2 / 3]))
        if rng.random() < 0.5:  # even sizes are the usual ones
            w, h = w & ~1, h & ~1
        step = rng.uniform(20.0, 32.0)
        f = (w / 2) / math.tan(math.radians(1.4 * step) / 2)
        rig = rng.choice(["tangent", "tangent", "cylinder"])
        if rig == "cylinder":
            cams = min(cams, 6)
            cw, ch = int(f * math.radians(step) * (cams - 1) + w * 1.02), int(h * 1.06)
        else:
            cw, ch = int(f * math.radians(step) * (cams - 1) + w) + 32, int(h * 1.2)
        if cw * ch <= most_px:
            return {"rig": rig, "cams": cams, "w": w, "h": h, "f": round(f, 3), "step": round(step, 3), "cw": cw, "ch": ch,
                    "levels": rng.randint(3, 6), "geo": rng.randint(0, 9999)}


def draw(rng):
    kind = rng.choice(["stitch", "stitch", "stitch", "stitch", "batch", "static", "host", "loss", "features", "features",
                       "match", "match", "register"])
    opts = {"seam": rng.random() < 0.3, "fp16": rng.random() < 0.25, "float": rng.random() < 0.35}
    if kind == "stitch":
        return {"kind": kind, **_draw_rig(rng, 60_000_000), **opts}
    if kind == "batch":
        return {"kind": kind, "rigs": rng.randint(2, 6), "geo": rng.randint(0, 9999), "most": rng.randint(0, 1),
                "fp16": opts["fp16"], "float": opts["float"]}
    if kind == "static":
        return {"kind": kind, **_draw_rig(rng, 400_000, 480), **opts, "fp16": False}
    if kind == "host":
        return {"kind": kind, **_draw_rig(rng, 10_000_000, 1920), **opts, "float": False}
    if kind == "loss":
        while True:
            c = _draw_rig(rng, 20_000_000, 2560)
            if c["rig"] == "tangent":
                return {"kind": kind, **c}
    if kind == "features":
        w = _log(rng, 320, 3840)
        return {"kind": kind, "w": w, "h": int(w * rng.choice([9 / 16, 3 / 4])), "points": _log(rng, 100, 2048),
                "areas": rng.randint(1, 3), "fast_t": rng.choice([10, 20, 30])}
    if kind == "match":
        return {"kind": kind, "points": _log(rng, 100, 2048), "tables": rng.randint(4, 16), "bits": rng.randint(10, 18),
                "iters": _log(rng, 100, 4096)}
    while True:
        c = _draw_rig(rng, 3_000_000, 1280)
        if c["rig"] == "tangent":
            return {"kind": kind, **c, "points": _log(rng, 200, 1000), "iters": _log(rng, 200, 1024)}


# ------------------------------------------------------------------------------------------------
# geometry and views


def _ry(deg):
    c, s = math.cos(math.radians(deg)), math.sin(math.radians(deg))
    return np.array([[c, 0.0, s], [0.0, 1.0, 0.0], [-s, 0.0, c]])


def _cameras(case):
    """(cameras, canvas) of a case's rig; canvas is None or (f, cx, cy) of a cylinder."""
    n, w, h, f, cw, ch = (case[k] for k in ("cams", "w", "h", "f", "cw", "ch"))
    K = np.array([[f, 0.0, (w - 1) / 2], [0.0, f, (h - 1) / 2], [0.0, 0.0, 1.0]])
    Ki, Kc = np.linalg.inv(K), np.diag([f, f, 1.0])
    yaws = [case["step"] * (i - (n - 1) / 2) for i in range(n)]
    if case["rig"] == "cylinder":
        return [Camera(w, h, K @ _ry(-y)) for y in yaws], (f, (cw - 1) / 2, (ch - 1) / 2)
    psi = np.random.default_rng(case["geo"]).uniform(-2.0, 2.0, n)
    out = []
    for i in range(n):
        tx, yaw = ((cw - 1) / 2, yaws[i]) if case["rig"] == "planar" else \
            ((cw - 1) / 2 + f * math.radians(yaws[i]), psi[i])
        M = np.array([[1.0, 0.0, tx], [0.0, 1.0, (ch - 1) / 2], [0.0, 0.0, 1.0]]) @ Kc @ _ry(yaw) @ Ki
        out.append(Camera(w, h, M / M[2, 2]))
    return out, None


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _scene(gen, w, h):
    """(1, 3, h, w) scene in [0, 255]: smooth noise of three scales and scattered hard-edged blocks."""
    img = torch.zeros((1, 3, h, w), device="cuda")
    for cell, amp in ((96, 110.0), (32, 70.0), (7, 30.0)):
        lat = torch.rand((1, 3, h // cell + 2, w // cell + 2), generator=gen, device="cuda") * amp
        img += F.interpolate(lat, size=(h, w), mode="bilinear", align_corners=True)
    for cell in (41, 13):
        gh, gw = h // cell + 1, w // cell + 1
        on = torch.rand((1, 1, gh, gw), generator=gen, device="cuda") < 0.2
        blk = torch.where(on, torch.rand((1, 3, gh, gw), generator=gen, device="cuda") * 160.0 - 80.0, 0.0)
        img += blk.repeat_interleave(cell, 2)[:, :, :h].repeat_interleave(cell, 3)[:, :, :, :w]
    return img.clamp_(0.0, 255.0)


def _views(case, cams, canvas, gen):
    """One (H, W, 3) uint8 CUDA frame per camera."""
    margin = 160
    sw, sh = case["cw"] + 2 * margin, case["ch"] + 2 * margin
    scene = _scene(gen, sw, sh)
    out = []
    for c in cams:
        v, u = torch.meshgrid(torch.arange(c.height, device="cuda", dtype=torch.float32),
                              torch.arange(c.width, device="cuda", dtype=torch.float32), indexing="ij")
        m = np.linalg.inv(c.H) if canvas else c.H
        p = [float(m[k, 0]) * u + float(m[k, 1]) * v + float(m[k, 2]) for k in range(3)]
        if canvas:
            x = canvas[0] * torch.atan2(p[0], p[2]) + canvas[1]
            y = canvas[0] * p[1] / torch.hypot(p[0], p[2]) + canvas[2]
        else:
            x, y = p[0] / p[2], p[1] / p[2]
        grid = torch.stack([(x + margin) * (2.0 / (sw - 1)) - 1.0, (y + margin) * (2.0 / (sh - 1)) - 1.0], -1)[None]
        img = F.grid_sample(scene, grid, mode="bilinear", padding_mode="reflection", align_corners=True)
        out.append(img[0].permute(1, 2, 0).round().clamp(0, 255).to(torch.uint8).contiguous())
    return out


def _batch_rigs(case):
    """The uneven rigs of a batch: 2 to 6 cameras of one resolution each, 20 to 30 degrees apart."""
    rng = np.random.default_rng(1000 + case["geo"])
    rigs = []
    for k in range(case["rigs"]):
        n = int(rng.integers(2, 7))
        w, h = [(1280, 720), (1920, 1080), (3840, 2160)][min(int(rng.integers(0, 3)), case["most"])]
        step, levels = float(rng.uniform(20.0, 30.0)), int(rng.integers(4, 7))
        f = (w / 2) / math.tan(math.radians(1.4 * step) / 2)
        rigs.append({"rig": "tangent", "cams": n, "w": w, "h": h, "f": f, "step": step, "levels": levels,
                     "cw": int(f * math.radians(step) * (n - 1) + w) + 33, "ch": h + 2 * int(round(0.1 * h)),
                     "geo": case["geo"] * 7919 + k})
    return rigs


def _rig(case, cams, canvas):
    return Rig(cams, case["cw"], case["ch"], case["levels"], band_fp16=case.get("fp16", False),
               out_float=case.get("float", False), weights="seam" if case.get("seam") else "feather", canvas=canvas)


def _params(case, cams, seed):
    """(N, 9) canvas-to-camera parameters and gains as refinement meets them: every camera but the
    first moved by up to 3 px at its corners, gains between 0.8 and 1.2."""
    rng = np.random.default_rng(seed)
    rows = []
    for i, c in enumerate(cams):
        src = np.array([[0.0, 0.0], [c.width - 1.0, 0.0], [c.width - 1.0, c.height - 1.0], [0.0, c.height - 1.0]])
        p = np.c_[src, np.ones(4)] @ c.H.T
        dst = p[:, :2] / p[:, 2:] + (rng.uniform(-3.0, 3.0, (4, 2)) if i else 0.0)
        M, r = [], []
        for (u, v), (x, y) in zip(src, dst):
            M += [[u, v, 1, 0, 0, 0, -u * x, -v * x], [0, 0, 0, u, v, 1, -u * y, -v * y]]
            r += [x, y]
        A = np.linalg.inv(np.append(np.linalg.solve(np.array(M), np.array(r)), 1.0).reshape(3, 3))
        rows.append(np.append((A / abs(A[2, 2])).reshape(9)[:8], rng.uniform(0.8, 1.2) if i else 1.0))
    return np.stack(rows)


def _pattern():
    return np.clip(np.rint(np.random.default_rng(0).normal(0.0, 31.0 / 5.0, (256, 4))), -15, 15).astype(np.int8)


def _bits(tables, bits):
    rng = np.random.default_rng(0)
    return np.stack([rng.choice(256, bits, replace=False) for _ in range(tables)]).astype(np.uint8)


def _words(seed, iters):
    return np.random.default_rng(seed).integers(0, 2 ** 32, (iters, 4), dtype=np.uint64).astype(np.uint32)


def _areas(case):
    """One area: the whole view; more: vertical strips of it, as overlaps with neighbours are."""
    w, h, n = case["w"], case["h"], case["areas"]
    return [(0, 0, w, h)] if n == 1 else [(k * w // n, 0, k * w // n + w // (n + 1), h) for k in range(n)]


def _features_pair(case, seed):
    """Descriptors and positions of two views: a third of the points appear in both, moved by a
    homography; descriptors cluster as those of real patches do and differ in a few bits."""
    rng = np.random.default_rng(seed)
    n = case["points"]
    base = rng.integers(0, 2, (24, 256))
    da = base[rng.integers(0, 24, n)] ^ (rng.random((n, 256)) < 0.22)
    db = base[rng.integers(0, 24, n)] ^ (rng.random((n, 256)) < 0.22)
    xa = np.stack([rng.integers(20, 3820, n), rng.integers(20, 2140, n)], 1)
    xb = np.stack([rng.integers(20, 3820, n), rng.integers(20, 2140, n)], 1)
    H = np.array([[1.02, 0.03, -900.0], [-0.02, 0.98, 35.0], [1.5e-5, -8e-6, 1.0]])
    both = rng.permutation(n)[: max(8, n // 3)]
    at = rng.permutation(n)[: len(both)]
    p = np.c_[xa[both], np.ones(len(both))] @ H.T
    xb[at] = np.rint(p[:, :2] / p[:, 2:] + rng.normal(0.0, 0.4, (len(both), 2)))
    db[at] = da[both] ^ (rng.random((len(both), 256)) < 0.04)
    pack = lambda d: np.packbits(d.astype(np.uint8), axis=1, bitorder="little")  # noqa: E731
    return xa.astype(np.int32), pack(da), xb.astype(np.int32), pack(db)


# ------------------------------------------------------------------------------------------------
# the cases


def _zeroed(ctx):
    """The context with its result tensors zero, so that what no call writes is defined."""
    for t in vars(ctx).values():
        if isinstance(t, torch.Tensor):
            t.zero_()
    return ctx


def prepare(case, seed):
    kind, gen = case["kind"], _generator(seed)
    s = {"kind": kind}
    if kind in ("stitch", "static", "host", "loss", "register"):
        cams, canvas = _cameras(case)
        s["frames"] = _views(case, cams, canvas, gen)
    if kind in ("stitch", "host", "loss"):
        s["rig"] = _rig(case, cams, canvas)
    if kind == "stitch":
        s["out"] = s["rig"].new_output()
    elif kind == "static":
        s["desc"] = stitch.make_desc(cams, case["cw"], case["ch"], case["levels"], out_float=case["float"],
                                     weights="seam" if case["seam"] else "feather", canvas=canvas)
        s["out"] = torch.empty((case["ch"], case["cw"], 3), dtype=torch.float32 if case["float"] else torch.uint8,
                               device="cuda")
    elif kind == "host":
        s["frames"] = [f.cpu().pin_memory() for f in s["frames"]]
        s["out"] = torch.zeros((case["ch"], case["cw"], 3), dtype=torch.uint8).pin_memory()
    elif kind == "loss":
        s["params"] = torch.from_numpy(_params(case, cams, seed)).cuda()
    elif kind == "batch":
        s["rigs"], s["frames"] = [], []
        for c in _batch_rigs(case):
            cams, canvas = _cameras(c)
            s["frames"].append(_views(c, cams, canvas, gen))
            s["rigs"].append(_rig({**c, "fp16": case["fp16"], "float": case["float"]}, cams, canvas))
        s["batch"] = Batch(s["rigs"])
        s["out"] = [r.new_output() for r in s["rigs"]]
    elif kind == "features":
        img = _scene(gen, case["w"], case["h"])
        s["frame"] = img[0].permute(1, 2, 0).round().to(torch.uint8).contiguous()
        s["areas"], s["pattern"], s["fast_t"] = _areas(case), _pattern(), case["fast_t"]
        s["lorb"] = _zeroed(LORB(case["w"], case["h"], case["points"]))
    elif kind == "match":
        s["args"] = [torch.from_numpy(t).cuda() for t in _features_pair(case, seed)]
        s["n"] = torch.tensor([case["points"]], dtype=torch.int32, device="cuda")
        s["bits"] = _bits(case["tables"], case["bits"])
        s["rnd"] = torch.from_numpy(_words(seed, case["iters"]).view(np.int32)).cuda()
        s["matcher"] = _zeroed(Matcher(case["points"], case["iters"]))
    elif kind == "register":
        w, h = case["w"], case["h"]
        s["areas"], s["pattern"], s["bits"] = ([(w // 2, 0, w, h)], [(0, 0, w // 2, h)]), _pattern(), _bits(8, 16)
        s["rnd"] = torch.from_numpy(_words(seed, case["iters"]).view(np.int32)).cuda()
        s["lorb"] = [_zeroed(LORB(w, h, case["points"])) for _ in range(2)]
        s["matcher"] = _zeroed(Matcher(case["points"], case["iters"]))
    return s


def run(s):
    kind = s["kind"]
    if kind == "stitch":
        return s["rig"].stitch(s["frames"], s["out"])
    if kind == "static":
        f, out = s["frames"], s["out"]
        stitch.stitch_frames_static(s["desc"][0], [t.data_ptr() for t in f], [t.stride(0) for t in f], out.data_ptr(),
                                    out.stride(0) * out.element_size(), torch.cuda.current_stream().cuda_stream)
        return out
    if kind == "host":
        return s["rig"].stitch_host_async(s["frames"], s["out"])
    if kind == "batch":
        return s["batch"].stitch(s["frames"], s["out"])
    if kind == "loss":
        return s["rig"].backward(s["frames"], s["params"])
    if kind == "features":
        return s["lorb"].detect(s["frame"], s["areas"], s["pattern"], s["fast_t"])
    if kind == "match":
        xa, da, xb, db = s["args"]
        return s["matcher"].match(xa, da, s["n"], xb, db, s["n"], s["bits"], s["rnd"])
    (xa, _, da, na), (xb, _, db, nb) = (c.detect(f, a, s["pattern"])
                                        for c, f, a in zip(s["lorb"], s["frames"], s["areas"]))
    return s["matcher"].match(xa, da, na, xb, db, nb, s["bits"], s["rnd"])


def work(case):
    """Inputs read once, outputs written once; operations of the definition of each step."""
    kind = case["kind"]
    if kind == "batch":
        parts = [work({"kind": "stitch", "float": case["float"], **c}) for c in _batch_rigs(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    if kind == "features":
        px = case["w"] * case["h"] if case["areas"] == 1 else case["h"] * sum(a[2] - a[0] for a in _areas(case))
        return {"bytes": 3 * px + 52 * case["points"], "flops": 60 * px}
    if kind == "match":
        n, t = case["points"], case["iters"]
        return {"bytes": 80 * n + 16 * t + 13 * n // 3, "flops": 600 * t + 30 * t * (n // 3)}
    src = case["cams"] * case["w"] * case["h"]
    px = case["cw"] * case["ch"]
    if kind == "register":
        return {"bytes": 3 * src // 2 + 80 * case["points"], "flops": 30 * src + 600 * case["iters"]}
    if kind == "loss":
        # only where at least two views overlap: about 30 % of every view
        return {"bytes": 3 * src * 3 // 10, "flops": 100 * src * 3 // 10}
    return {"bytes": 3 * src + (12 if case.get("float") else 3) * px, "flops": 130 * src + 35 * px}


# ------------------------------------------------------------------------------------------------
# the same results in 64 bits


def exact(case, seed):
    kind = case["kind"]
    if kind in ("stitch", "static") and case["float"] and case["cams"] * case["cw"] * case["ch"] <= 500_000_000:
        cams, canvas = _cameras(case)
        frames = _views(case, cams, canvas, _generator(seed))
        return _exact_canvas(case, cams, canvas, frames)
    if kind == "loss":
        cams, canvas = _cameras(case)
        return _exact_loss(case, _views(case, cams, canvas, _generator(seed)), _params(case, cams, seed))
    if kind == "match":
        xa, da, xb, db = _features_pair(case, seed)
        return _exact_match(xa, da, xb, db, _bits(case["tables"], case["bits"]), _words(seed, case["iters"]))
    if kind == "register" and case["w"] <= 800:
        cams, canvas = _cameras(case)
        fa, fb = _views(case, cams, canvas, _generator(seed))[:2]
        w, h, n = case["w"], case["h"], case["points"]
        xa, da = _exact_features(fa, (w // 2, 0, w, h), n)
        xb, db = _exact_features(fb, (0, 0, w // 2, h), n)
        return _exact_match(xa, da, xb, db, _bits(8, 16), _words(seed, case["iters"]))
    return None


def _fold(i, n):
    if n == 1:
        return torch.zeros_like(i)
    i = i.abs() % (2 * n - 2)
    return torch.where(i < n, i, 2 * n - 2 - i)


def _reduce(t):
    for d in (0, 1):
        n = t.shape[d]
        k = 2 * torch.arange((n + 1) // 2, device=t.device)
        t = sum(wt * t.index_select(d, _fold(k + o, n)) for o, wt in zip(range(-2, 3), (1 / 16, 1 / 4, 3 / 8, 1 / 4, 1 / 16)))
    return t


def _expand(t, h, w):
    for d, size in ((0, h), (1, w)):
        n = t.shape[d]
        x = torch.arange(size, device=t.device)
        at = lambda o: t.index_select(d, _fold(torch.div(x, 2, rounding_mode="floor") + o, n))  # noqa: E731
        odd = (x % 2 == 1).reshape([-1 if k == d else 1 for k in range(t.dim())])
        t = torch.where(odd, 0.5 * (at(0) + at(1)), 0.75 * at(0) + 0.125 * (at(-1) + at(1)))
    return t


def _bilinear(frame, u, v):
    """Bilinear sample with clamped coordinates of an (H, W, 3) float64 frame."""
    h, w = frame.shape[:2]
    u, v = u.clamp(0, w - 1), v.clamp(0, h - 1)
    i, j = u.detach().floor().long(), v.detach().floor().long()
    fx, fy = (u - i)[..., None], (v - j)[..., None]
    i1, j1 = (i + 1).clamp(max=w - 1), (j + 1).clamp(max=h - 1)
    top = frame[j, i] + fx * (frame[j, i1] - frame[j, i])
    bot = frame[j1, i] + fx * (frame[j1, i1] - frame[j1, i])
    return top + fy * (bot - top)


def _exact_canvas(case, cams, canvas, frames):
    cw, ch = case["cw"], case["ch"]
    y, x = torch.meshgrid(torch.arange(ch, device="cuda", dtype=torch.float64),
                          torch.arange(cw, device="cuda", dtype=torch.float64), indexing="ij")
    if canvas:
        f, cx, cy = canvas
        ray = (torch.sin((x - cx) / f), (y - cy) / f, torch.cos((x - cx) / f))
    else:
        ray = (x, y, torch.ones_like(x))
    images, feather = [], []
    for c, fr in zip(cams, frames):
        A = c.H if canvas else np.linalg.inv(c.H)
        if not canvas:
            A = A / abs(A[2, 2])
        p = [float(A[k, 0]) * ray[0] + float(A[k, 1]) * ray[1] + float(A[k, 2]) * ray[2] for k in range(3)]
        u, v = p[0] / p[2], p[1] / p[2]
        W, H = c.width, c.height
        ok = (p[2] > 0) & (u >= -0.5) & (u < W - 0.5) & (v >= -0.5) & (v < H - 0.5)
        m = torch.minimum(torch.minimum(u + 0.5, v + 0.5), torch.minimum(W - 0.5 - u, H - 0.5 - v))
        feather.append(torch.where(ok, m.clamp(min=0.0), 0.0))
        u, v = torch.nan_to_num(u), torch.nan_to_num(v)
        img = _bilinear(fr.double(), u, v) * (c.gain / 255.0)
        images.append(torch.where((p[2] > 0)[..., None], img, 0.0))
    total = sum(feather)
    if case["seam"]:
        wmax, taken = torch.stack(feather).amax(0), torch.zeros_like(total, dtype=torch.bool)
        weights = []
        for w in feather:
            own = (w > 0) & (w >= (1 - 1e-9) * wmax) & ~taken
            taken |= own
            weights.append(own.double())
    else:
        weights = [torch.where(total > 0, w / total, 0.0) for w in feather]
    L = case["levels"]
    shapes = [(ch, cw)]
    for _ in range(L - 1):
        shapes.append(((shapes[-1][0] + 1) // 2, (shapes[-1][1] + 1) // 2))
    num = [torch.zeros((*sh, 3), device="cuda", dtype=torch.float64) for sh in shapes]
    den = [torch.zeros((*sh, 1), device="cuda", dtype=torch.float64) for sh in shapes]
    for g, w in zip(images, weights):
        w = w[..., None]
        for lv in range(L):
            nxt = _reduce(g) if lv + 1 < L else None
            num[lv] += w * (g - _expand(nxt, *shapes[lv]) if nxt is not None else g)
            den[lv] += w
            g, w = nxt, _reduce(w) if nxt is not None else None
    out = None
    for lv in reversed(range(L)):
        band = torch.where(den[lv] > 1e-12, num[lv] / den[lv].clamp(min=1e-300), 0.0)
        out = band if out is None else band + _expand(out, *shapes[lv])
    return torch.where((total > 0)[..., None], out.clamp(0.0, 1.0), 0.0)


def _exact_loss(case, frames, params):
    par = torch.from_numpy(params).cuda().requires_grad_(True)
    cams, _ = _cameras(case)
    sign = [1.0 if np.linalg.inv(c.H)[2, 2] > 0 else -1.0 for c in cams]
    frames = [f.double() / 255.0 for f in frames]
    total = torch.zeros((), device="cuda", dtype=torch.float64)
    x = torch.arange(case["cw"], device="cuda", dtype=torch.float64)
    for y0 in range(0, case["ch"], 128):
        y = torch.arange(y0, min(y0 + 128, case["ch"]), device="cuda", dtype=torch.float64)[:, None]
        valid, img = [], []
        for k, fr in enumerate(frames):
            a = par[k]
            w = a[6] * x + a[7] * y + sign[k]
            u, v = (a[0] * x + a[1] * y + a[2]) / w, (a[3] * x + a[4] * y + a[5]) / w
            h, wd = fr.shape[:2]
            valid.append(((w > 0) & (u >= -0.5) & (u < wd - 0.5) & (v >= -0.5) & (v < h - 0.5)).detach())
            ok = valid[-1]
            img.append(a[8] * _bilinear(fr, torch.where(ok, u, 0.0), torch.where(ok, v, 0.0)))
        loss = sum((((img[i] - img[j]) ** 2).sum(-1) * (valid[i] & valid[j])).sum()
                   for i in range(len(img)) for j in range(i + 1, len(img)))
        loss.backward()
        total += loss.detach()
    return total.reshape(1), par.grad


def _exact_features(frame, area, n):
    """L-ORB of one area: positions and descriptors of the n strongest corners (FAST threshold 20)."""
    px = frame.cpu().numpy().astype(np.int64)
    g = (77 * px[..., 0] + 150 * px[..., 1] + 29 * px[..., 2] + 128) >> 8
    h, w = g.shape
    sh = lambda a, dx, dy: np.roll(a, (-dy, -dx), (0, 1))  # a at (x + dx, y + dy)  # noqa: E731
    ring = [(0, -3), (1, -3), (2, -2), (3, -1), (3, 0), (3, 1), (2, 2), (1, 3), (0, 3), (-1, 3), (-2, 2), (-3, 1),
            (-3, 0), (-3, -1), (-2, -2), (-1, -3)]
    corner = np.zeros((h, w), bool)
    for sgn in (1, -1):
        t = np.stack([sgn * (sh(g, dx, dy) - g) > 20 for dx, dy in ring])
        for k in range(16):
            corner |= np.logical_and.reduce([t[(k + m) % 16] for m in range(9)])
    ix, iy = sh(g, 1, 0) - sh(g, -1, 0), sh(g, 0, 1) - sh(g, 0, -1)
    k5 = (1, 4, 6, 4, 1)

    def smooth(a):
        a = sum(wt * sh(a, o, 0) for o, wt in zip(range(-2, 3), k5))
        return sum(wt * sh(a, 0, o) for o, wt in zip(range(-2, 3), k5))

    A, B, C = smooth(ix * ix), smooth(iy * iy), smooth(ix * iy)
    R = 25 * (A * B - C * C) - (A + B) ** 2
    box = np.zeros((h, w), bool)
    box[max(area[1], 18):min(area[3], h - 18), max(area[0], 18):min(area[2], w - 18)] = True
    low = np.iinfo(np.int64).min
    R = np.where(corner & box & (R > 0), R, low)
    keep = R != low
    for dy in (-1, 0, 1):
        for dx in (-1, 0, 1):
            if dx or dy:
                o = sh(R, dx, dy)
                keep &= (R > o) | ((R == o) & ((dy, dx) > (0, 0))) | (o == low)
    ys, xs = np.nonzero(keep)
    order = np.lexsort((ys * w + xs, -R[ys, xs]))[:n]
    ys, xs = ys[order], xs[order]
    S, p = smooth(g), _pattern().astype(np.int64)
    d = S[ys[:, None] + p[:, 1], xs[:, None] + p[:, 0]] > S[ys[:, None] + p[:, 3], xs[:, None] + p[:, 2]]
    return np.stack([xs, ys], 1), np.packbits(d.astype(np.uint8), axis=1, bitorder="little")


def _exact_match(xa, da, xb, db, bits, words):
    """The homography alone (the other outputs are whole numbers)."""
    nothing = (None, None, np.eye(3).reshape(9), None, None)
    ua, ub = (np.unpackbits(d, axis=1, bitorder="little").astype(np.int64) for d in (da, db))
    probed = np.zeros((len(ua), len(ub)), bool)
    for t in bits:
        probed |= (ua[:, None, t] != ub[None, :, t]).sum(-1) <= 1
    dist = np.where(probed, ua @ (1 - ub).T + (1 - ua) @ ub.T, 1 << 20)
    rows = np.arange(len(ua))
    b1 = dist.argmin(1)
    d1 = dist[rows, b1]
    rest = dist.copy()
    rest[rows, b1] = 1 << 20
    d2 = rest.min(1)
    ok = (d1 <= 80) & ((d2 >= 1 << 20) | (5 * d1 < 4 * d2))
    a = rows[ok][np.lexsort((rows[ok], d1[ok]))]
    n = len(a)
    if n < 4:
        return nothing
    pa, pb = xa[a].astype(np.float64), xb[b1[a]].astype(np.float64)
    ca, cb = (0.5 * (p.min(0) + p.max(0)) for p in (pa, pb))
    sa, sb = (2.0 / max(np.ptp(p, axis=0).max(), 1.0) for p in (pa, pb))
    qa, qb = (pa - ca) * sa, (pb - cb) * sb
    M = np.zeros((n, 2, 8))
    M[:, 0, :2], M[:, 0, 2], M[:, 1, 3:5], M[:, 1, 5] = qa, 1.0, qa, 1.0
    M[:, :, 6:] = -qb[:, :, None] * qa[:, None, :]
    grow, q = [1], n * (n - 1) * (n - 2) * (n - 3)
    for m in range(4, n):
        grow.append(grow[-1] + -(-800000 * m * (m - 1) * (m - 2) // q))
    best, best_h = -1, None
    for t in range(1, len(words) + 1):
        c = int(np.searchsorted(grow[:n - 4], t, side="right"))
        top, picked = 4 + c, []
        uniform = grow[c] < t
        pool = top if uniform else top - 1
        for k in range(4 if uniform else 3):
            j = int(words[t - 1, k]) % (pool - k)
            for taken in sorted(picked):
                j += taken <= j
            picked.append(j)
        at = picked if uniform else [top - 1] + picked
        sys8, rhs = M[at].reshape(8, 8), qb[at].reshape(8)
        if np.linalg.matrix_rank(sys8, tol=1e-11) < 8:
            continue
        hyp = np.append(np.linalg.solve(sys8, rhs), 1.0).reshape(3, 3)
        p = np.c_[qa, np.ones(n)] @ hyp.T
        with np.errstate(all="ignore"):
            inl = (p[:, 2] > 0) & (((p[:, :2] / p[:, 2:] - qb) ** 2).sum(1) < (3.0 * sb) ** 2)
        if inl.sum() > best:
            best, best_h = int(inl.sum()), inl
    if best < 4:
        return nothing
    h = np.append(np.linalg.lstsq(M[best_h].reshape(-1, 8), qb[best_h].reshape(-1), rcond=None)[0], 1.0).reshape(3, 3)
    Ta = np.array([[sa, 0, -sa * ca[0]], [0, sa, -sa * ca[1]], [0, 0, 1]])
    Tb = np.array([[1 / sb, 0, cb[0]], [0, 1 / sb, cb[1]], [0, 0, 1]])
    H = Tb @ h @ Ta
    return None, None, (H / H[2, 2]).reshape(9), None, None
