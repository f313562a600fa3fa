"""The work a renderer gives this library, as measurable cases: whole frames of one view from 64x64
to 4K, many views per frame, the temporal path with and without the tile cache and the probe filter,
the world cache alone on ragged batches, the probe filter alone, and the learned surrogate (training,
far-hit queries, inference of points).

Every case runs through the package's public entry points on device buffers.  Inputs are made on the
GPU from a seed: a room of axis-aligned boxes or a Cornell box (the scenes of this repository's
configurations, with fewer boxes so that tracing them is quick), its G-buffer, and one frame's probe
rays traced against it.  A state holds two consecutive frames, which its passes take in turn with a
growing frame index, and a cache that has already resolved a frame."""
import math

import numpy as np
import torch

import paper_2310_19855_gb300 as gi
from paper_2310_19855_gb300.pipeline import BatchPipeline, Pipeline, TemporalPipeline

DEV = "cuda"
FOV = math.radians(60.0)
CELL, ALPHA, LODS = 0.05, 0.1, 4
CORNELL_AABB = ((-1.05, -0.05, -1.05), (1.05, 2.05, 1.05))
ROOM = (64.0, 16.0, 64.0)
VIEW_SIZES = ((640, 360), (1280, 720), (1920, 1080), (2560, 1440))


def listed():
    return [
        # the smallest call: a 64x64 preview (or a probe-lighting thumbnail), 4 rays per cell; launch latency counts
        {"name": "frame_cornell_64", "kind": "frame", "scene": "cornell", "width": 64, "height": 64, "rpp": 256,
         "log2_slots": 16, "key_dir": 0, "f16": False, "first_touch": 0},
        # one game frame at 1080p: the library's ordinary use
        {"name": "frame_boxes_1080p", "kind": "frame", "scene": "boxes", "width": 1920, "height": 1080, "rpp": 64,
         "log2_slots": 22, "key_dir": 0, "f16": False, "first_touch": 0},
        # a 4K frame with half-precision storage of the resolved radiance: the largest table and most records
        {"name": "frame_boxes_4k_f16", "kind": "frame", "scene": "boxes", "width": 3840, "height": 2160, "rpp": 64,
         "log2_slots": 24, "key_dir": 0, "f16": True, "first_touch": 0},
        # an editor viewport of odd size, ray-direction descriptor, two rays per cell, touch list
        {"name": "frame_odd_ray_list", "kind": "frame", "scene": "boxes", "width": 1283, "height": 717, "rpp": 128,
         "log2_slots": 21, "key_dir": 1, "f16": False, "first_touch": 1},
        # a render farm's node or split-screen server: 16 views of uneven size, one launch per pass, replayed graph
        {"name": "batch_16_views", "kind": "batch", "views": 16, "size_pick": 0, "graph": True},
        # the quarter-sample operating point: 2x2 temporal upscale, reprojection, hysteresis
        {"name": "temporal_1080p", "kind": "temporal", "width": 1920, "height": 1080, "rpp": 64, "upscale": 2,
         "log2_slots": 22, "tiles": False, "filtered": False},
        # the whole chain at that point: two-level tile cache and probe filter
        {"name": "chain_tiles_filter_1080p", "kind": "temporal", "width": 1920, "height": 1080, "rpp": 64, "upscale": 2,
         "log2_slots": 18, "tiles": True, "filtered": True},
        # the cache by itself, as another light-transport code uses it: a ragged batch, answers by slot and by point
        {"name": "cache_ragged", "kind": "cache", "n": 777777, "log2_slots": 21, "key_dir": 0, "f16": False,
         "first_touch": 0, "merge": 0, "tiles": False},
        # the filtered probe stage of a full-rate 1080p frame
        {"name": "probe_filter_1080p", "kind": "filter", "width": 1920, "height": 1080, "rpp": 64, "log2_slots": 22},
        # the surrogate's training of one frame: 65,536 samples in four Adam steps
        {"name": "surrogate_train", "kind": "train", "width": 1920, "height": 1080, "log2_table": 19, "batch": 65536,
         "steps": 4},
        # a frame whose far hits are answered by the network
        {"name": "surrogate_far_1080p", "kind": "far", "width": 1920, "height": 1080, "rpp": 64, "log2_slots": 22,
         "log2_table": 19},
        # radiance of arbitrary points (light-map texels, volume samples) from the network
        {"name": "surrogate_infer", "kind": "infer", "n": 100003, "log2_table": 19},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo, hi):
    h = _log_int(rng, lo, hi)
    return max(16, int(h * rng.choice((1.0, 4 / 3, 16 / 9, 21 / 9))) + rng.randint(0, 9)), h


def _slots(n):
    """Table of at least twice as many slots as a frame has records, as the configurations have."""
    return min(25, max(14, int(math.ceil(math.log2(max(n, 1)))) + 1))


def draw(rng):
    kind = rng.choice(("frame", "frame", "temporal", "cache", "batch", "filter", "train", "far", "infer"))
    if kind == "frame":
        w, h = _size(rng, 64, 1600)
        rpp = rng.choice((64, 64, 64, 128, 256)) if w * h < 1_500_000 else 64
        n = ((w + 7) // 8) * ((h + 7) // 8) * rpp
        return {"kind": kind, "scene": rng.choice(("cornell", "boxes")), "width": w, "height": h, "rpp": rpp,
                "log2_slots": _slots(n), "key_dir": rng.choice((0, 0, 1)), "f16": rng.random() < 0.3,
                "first_touch": rng.choice((0, 0, 1, 2))}
    if kind == "temporal":
        w, h = _size(rng, 180, 1440)
        u, tiles = rng.choice((1, 2, 2, 3)), rng.random() < 0.5
        n = (w // (8 * u) + 1) * (h // (8 * u) + 1) * 64
        return {"kind": kind, "width": w, "height": h, "rpp": 64, "upscale": u,
                "log2_slots": max(12, _slots(n) - 3) if tiles else _slots(n), "tiles": tiles,
                "filtered": rng.random() < 0.5}
    if kind == "cache":
        n, tiles = _log_int(rng, 1000, 4_000_000), rng.random() < 0.3
        return {"kind": kind, "n": n, "log2_slots": max(12, _slots(n) - 3) if tiles else _slots(n),
                "key_dir": rng.choice((0, 1)), "f16": rng.random() < 0.3,
                "first_touch": 0 if tiles else rng.choice((0, 0, 1)), "merge": 0 if tiles else rng.choice((0, 0, 1)),
                "tiles": tiles}
    if kind == "batch":
        return {"kind": kind, "views": rng.randint(2, 12), "size_pick": rng.randint(1, 10 ** 6), "graph": rng.random() < 0.7}
    if kind == "filter":
        w, h = _size(rng, 180, 1440)
        rpp = rng.choice((64, 64, 128))
        return {"kind": kind, "width": w, "height": h, "rpp": rpp,
                "log2_slots": _slots(((w + 7) // 8) * ((h + 7) // 8) * rpp)}
    if kind == "train":
        w, h = _size(rng, 256, 1080)
        steps = rng.choice((1, 2, 4))
        return {"kind": kind, "width": w, "height": h, "log2_table": rng.randint(15, 19),
                "batch": steps * _log_int(rng, 2048, 32768), "steps": steps}
    if kind == "far":
        w, h = _size(rng, 360, 1080)
        return {"kind": kind, "width": w, "height": h, "rpp": 64, "log2_slots": 21, "log2_table": rng.randint(15, 19)}
    return {"kind": kind, "n": _log_int(rng, 300, 1_000_000), "log2_table": rng.randint(14, 19)}


# ---------------------------------------------------------------------------------------- scenes

def _scene(kind, g):
    """Boxes (lo, hi), albedo, emission, light position and intensity on the device."""
    def rand(*s, lo=0.0, hi=1.0):
        return torch.rand(*s, generator=g, device=DEV) * (hi - lo) + lo

    w = 0.05
    if kind == "cornell":
        j = rand(4, lo=-0.1, hi=0.1).tolist()
        b = [((-1 - w, -w, -1 - w), (1 + w, 0, 1 + w)), ((-1 - w, 2, -1 - w), (1 + w, 2 + w, 1 + w)),
             ((-1 - w, -w, -1 - w), (1 + w, 2 + w, -1)), ((-1 - w, -w, -1 - w), (-1, 2 + w, 1 + w)),
             ((1, -w, -1 - w), (1 + w, 2 + w, 1 + w)),
             ((-0.65 + j[0], 0, j[1]), (-0.05 + j[0], 0.6, 0.6 + j[1])),
             ((0.05 + j[2], 0, -0.6 + j[3]), (0.65 + j[2], 1.2, j[3])), ((-0.25, 1.98, -0.25), (0.25, 2.0, 0.25))]
        lo, hi = (torch.tensor([x[k] for x in b], device=DEV, dtype=torch.float32) for k in (0, 1))
        emit = torch.zeros(len(b), 3, device=DEV)
        emit[-1] = torch.tensor((10.0, 9.0, 7.5), device=DEV)
        light, power = (0.0, 1.85, 0.0), (3.0, 3.0, 3.0)
    else:
        lx, ly, lz = ROOM if kind == "boxes" else (24.0, 8.0, 24.0)
        nb = 1018 if kind == "boxes" else 250
        w = 0.2
        b = [((-w, -w, -w), (lx + w, 0, lz + w)), ((-w, ly, -w), (lx + w, ly + w, lz + w)),
             ((-w, -w, -w), (0, ly + w, lz + w)), ((lx, -w, -w), (lx + w, ly + w, lz + w)),
             ((-w, -w, -w), (lx + w, ly + w, 0)), ((-w, -w, lz), (lx + w, ly + w, lz + w))]
        c = torch.rand(nb, 3, generator=g, device=DEV) * torch.tensor((lx, ly, lz), device=DEV)
        s = 0.1 * torch.pow(50.0, torch.rand(nb, 3, generator=g, device=DEV))  # half sizes of 0.05 .. 2.5 m
        lo, hi = (torch.tensor([x[k] for x in b], device=DEV, dtype=torch.float32) for k in (0, 1))
        lo, hi = torch.cat((lo, c - 0.5 * s)), torch.cat((hi, c + 0.5 * s))
        emit = torch.where(torch.rand(nb + 6, 1, generator=g, device=DEV) < 0.02, rand(nb + 6, 3, lo=1, hi=50),
                           torch.zeros((), device=DEV))
        emit[:6] = 0
        light, power = (0.7 * lx, 0.75 * ly, 0.5 * lz), (2000.0, 1800.0, 1600.0)
    return {"kind": kind, "lo": lo, "hi": hi, "albedo": rand(lo.shape[0], 3, lo=0.2, hi=0.8), "emit": emit,
            "light": torch.tensor(light, device=DEV), "power": torch.tensor(power, device=DEV),
            "room": (2.0, 2.0, 2.0) if kind == "cornell" else (lx, ly, lz), "turn": float(rand(1))}


def _trace(sc, o, d):
    """Closest box of each ray (n, 3): distance (inf for none), box, unit face normal."""
    n, B = o.shape[0], sc["lo"].shape[0]
    t, box = torch.empty(n, device=DEV), torch.empty(n, dtype=torch.int64, device=DEV)
    inv = 1.0 / torch.where(d.abs() < 1e-12, torch.full((), 1e-12, device=DEV), d)
    step = max(1, (1 << 23) // B)
    for i in range(0, n, step):
        near = far = None
        for a in range(3):
            oa, ia = o[i:i + step, a, None], inv[i:i + step, a, None]
            p, q = (sc["lo"][None, :, a] - oa).mul_(ia), (sc["hi"][None, :, a] - oa).mul_(ia)
            lo_, hi_ = torch.minimum(p, q), torch.maximum(p, q)
            near = lo_ if near is None else torch.maximum(near, lo_, out=near)
            far = hi_ if far is None else torch.minimum(far, hi_, out=far)
        near.masked_fill_((far < near) | (near < 1e-4), math.inf)
        t[i:i + step], box[i:i + step] = near.min(dim=1)
    lo, hi = sc["lo"][box], sc["hi"][box]
    per = torch.minimum((lo - o) * inv, (hi - o) * inv)
    axis = per.argmax(dim=1, keepdim=True)
    nrm = torch.zeros(n, 3, device=DEV).scatter_(1, axis, -torch.sign(d.gather(1, axis)))
    nrm = torch.where(torch.isfinite(t)[:, None], nrm, torch.zeros((), device=DEV))
    return t, box, nrm


class _Cam:
    """Pinhole camera; also what view_of() takes."""

    def __init__(self, sc, f, width, height):
        if sc["kind"] == "cornell":
            pos, fwd = np.array((0.02 * f, 1.0, 2.6)), np.array((0.0, 0.0, -1.0))
        else:
            a = 2 * math.pi * sc["turn"]
            lx, ly, lz = sc["room"]
            pos = np.array((0.5 * lx + 0.25 * lx * math.cos(a), 0.35 * ly, 0.5 * lz + 0.25 * lz * math.sin(a)))
            fwd = np.array((-math.cos(a + 0.4), -0.05, -math.sin(a + 0.4)))
            pos = pos + 0.08 * f * fwd
        fwd = fwd / np.linalg.norm(fwd)
        right = np.cross(fwd, (0.0, 1.0, 0.0))
        right /= np.linalg.norm(right)
        up = np.cross(right, fwd)
        self.pos, self.fwd, self.right, self.up = (v.astype(np.float32) for v in (pos, fwd, right, up))
        self.fov_y, self.width, self.height = FOV, width, height

    def view(self, frame):
        return gi.make_view(frame, self.width, self.height, self.pos, self.fwd, self.right, self.up, self.fov_y)

    def rays(self, xs, ys, dtype=torch.float32):
        """Unit directions through pixel centres."""
        th = math.tan(0.5 * self.fov_y)
        sx = (2 * (xs.to(dtype) + 0.5) / self.width - 1) * (th * self.width / self.height)
        sy = (1 - 2 * (ys.to(dtype) + 0.5) / self.height) * th
        f, r, u = (torch.tensor(v, device=DEV).to(dtype) for v in (self.fwd, self.right, self.up))
        d = f + sx[..., None] * r + sy[..., None] * u
        return d / d.norm(dim=-1, keepdim=True)


def _halton(i, base, scale):
    num, den = 0, 1
    while i:
        num, den, i = num * base + i % base, den * base, i // base
    return scale * num // den


def _frame_basis(n):
    """Tangent and bitangent of unit normals (Duff et al. 2017)."""
    s = torch.where(torch.signbit(n[..., 2]), -torch.ones_like(n[..., 2]), torch.ones_like(n[..., 2]))
    a = -1.0 / (s + n[..., 2])
    b = n[..., 0] * n[..., 1] * a
    t = torch.stack((1 + s * n[..., 0] ** 2 * a, s * b, -s * n[..., 0]), -1)
    return t, torch.stack((b, s + n[..., 1] ** 2 * a, -n[..., 1]), -1)


def _pixels(w, h):
    return torch.meshgrid(torch.arange(h, device=DEV), torch.arange(w, device=DEV), indexing="ij")


def _frame(sc, f, w, h, rpp, g, upscale=1, jitter_frame=None, prev=None):
    """Frame f: camera, G-buffer (h, w, 4), records (13, R) of the spawn tiles' probes, motion vectors."""
    cam = _Cam(sc, f, w, h)
    ys, xs = _pixels(w, h)
    d = cam.rays(xs, ys).reshape(-1, 3)
    o = torch.tensor(cam.pos, device=DEV)
    t, _, nrm = _trace(sc, o.expand(d.shape[0], 3), d)
    gbuf = torch.cat((nrm, t[:, None]), 1).reshape(h, w, 4).contiguous()
    jf, st = (f if jitter_frame is None else jitter_frame) + 1, 8 * upscale
    ty, tx = torch.meshgrid(torch.arange(-(-h // st), device=DEV), torch.arange(-(-w // st), device=DEV), indexing="ij")
    px = (st * tx + _halton(jf, 2, st)).clamp(max=w - 1).reshape(-1)
    py = (st * ty + _halton(jf, 3, st)).clamp(max=h - 1).reshape(-1)
    pn = gbuf[py, px]
    valid = torch.isfinite(pn[:, 3])
    n = torch.where(valid[:, None], pn[:, :3], torch.tensor((0.0, 0.0, 1.0), device=DEV))
    at = o + cam.rays(px, py) * torch.where(valid, pn[:, 3], torch.zeros((), device=DEV))[:, None] + 1e-3 * n
    P = px.numel()
    cell = torch.arange(rpp, device=DEV) % 64
    ab = torch.rand(P, rpp, 2, generator=g, device=DEV)
    u, v = -1 + (cell % 8 + ab[..., 0]) * 0.25, -1 + (cell // 8 + ab[..., 1]) * 0.25
    x, y = 0.5 * (u + v), 0.5 * (u - v)
    l3 = torch.stack((x, y, 1 - x.abs() - y.abs()), -1)
    l3 = l3 / l3.norm(dim=-1, keepdim=True)
    tb, bb = _frame_basis(n)
    rd = (l3[..., 0:1] * tb[:, None] + l3[..., 1:2] * bb[:, None] + l3[..., 2:3] * n[:, None]).reshape(-1, 3)
    ro = at[:, None].expand(P, rpp, 3).reshape(-1, 3)
    t, box, rn = _trace(sc, ro, rd)
    live = valid.repeat_interleave(rpp)
    hit = torch.isfinite(t) & live
    pos = torch.where(hit[:, None], ro + rd * torch.where(hit, t, torch.zeros((), device=DEV))[:, None], torch.zeros((), device=DEV))
    rn = torch.where(hit[:, None], rn, torch.zeros((), device=DEV))
    to = sc["light"] - pos
    r2 = (to * to).sum(1)
    irr = ((to * rn).sum(1) / r2.sqrt().clamp(min=1e-6)).clamp(min=0) / r2.clamp(min=1e-4)
    rad = sc["albedo"][box] / math.pi * irr[:, None] * sc["power"] + sc["emit"][box]
    rad = torch.where(hit[:, None], rad + 0.05 * torch.rand(rad.shape, generator=g, device=DEV), torch.zeros((), device=DEV))
    ln = torch.where(hit, t, torch.full((), math.inf, device=DEV))
    ln = torch.where(live, ln, -torch.ones((), device=DEV))
    rec = torch.cat((pos.T, rn.T, rad.T, ln[None], rd.T)).contiguous()
    motion = None
    if prev is not None:
        p = o.double() + cam.rays(xs, ys, torch.float64) * torch.where(torch.isfinite(gbuf[..., 3]), gbuf[..., 3], torch.zeros((), device=DEV)).double()[..., None]
        q = p - torch.tensor(prev.pos, device=DEV).double()
        z, a, b = (q @ torch.tensor(v, device=DEV).double() for v in (prev.fwd, prev.right, prev.up))
        th = math.tan(0.5 * FOV)
        ok = torch.isfinite(gbuf[..., 3]) & (z > 0)
        mx = (a / (z * th * w / h) + 1) * 0.5 * w - (xs + 0.5)
        my = (1 - b / (z * th)) * 0.5 * h - (ys + 0.5)
        motion = torch.where(ok[..., None], torch.stack((mx, my), -1), torch.zeros((), device=DEV).double()).float().contiguous()
    return {"cam": cam, "gbuf": gbuf, "rec": rec, "motion": motion, "index": f}


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _two(case, seed):
    """The scene and two consecutive frames of a single-view case."""
    g = _gen(seed)
    sc = _scene(case.get("scene", "boxes"), g)
    return [_frame(sc, f, case["width"], case["height"], case["rpp"], g) for f in (0, 1)]


def _batch_views(case):
    """(scene, width, height, log2_slots) of each view: Cornell boxes and small rooms in turn."""
    out = []
    r = np.random.RandomState(case["size_pick"])
    for v in range(case["views"]):
        w, h = VIEW_SIZES[v % 4] if case["size_pick"] == 0 else (int(r.randint(100, 1700)), int(r.randint(90, 1000)))
        out.append(("cornell" if v % 2 == 0 else "room", w, h, 21 if w * h > 1_000_000 else 20))
    return out


def _batch_frames(case, seed):
    per = []
    for v, (scene, w, h, _) in enumerate(_batch_views(case)):
        g = _gen(seed * 1000 + v)
        sc = _scene(scene, g)
        per.append([_frame(sc, f, w, h, 64, g) for f in (0, 1)])
    return per


def _cache_frames(case, seed):
    """Records of two frames cut to n."""
    n = case["n"]
    side = 8 * math.ceil(math.sqrt(n / 64))
    g = _gen(seed)
    sc = _scene("boxes", g)
    return [dict(f, rec=f["rec"][:, :n].contiguous()) for f in (_frame(sc, k, side, side, 64, g) for k in (0, 1))]


def _infer_inputs(case, seed):
    g = _gen(seed)
    T, n = 1 << case["log2_table"], case["n"]

    def uni(*s):
        return torch.rand(*s, generator=g, device=DEV) * 2 - 1

    prm = (0.5 * uni(16, T, 2), math.sqrt(6 / 96) * uni(64, 32), math.sqrt(6 / 128) * uni(64, 64), math.sqrt(6 / 67) * uni(3, 64))
    lo, hi = (torch.tensor(v, device=DEV) for v in CORNELL_AABB)
    # points on the box's surfaces' scale: uniform in it, axis-aligned normals
    pos = (lo[:, None] + (hi - lo)[:, None] * (0.5 + 0.49 * uni(3, n))).contiguous()
    ax = torch.randint(0, 3, (n,), generator=g, device=DEV)
    nrm = torch.zeros(3, n, device=DEV)
    nrm[ax, torch.arange(n, device=DEV)] = torch.sign(uni(n)) + 0.0
    return prm, pos, nrm


# ---------------------------------------------------------------------------------------- cases

def prepare(case, seed):
    kind = case["kind"]
    if kind in ("frame", "filter"):
        fr = _two(case, seed)
        pl = Pipeline(case["width"], case["height"], case["rpp"], case["log2_slots"], key_dir=case.get("key_dir", 0),
                      resolved_format=int(case.get("f16", False)), first_touch=case.get("first_touch", 0))
        s = {"case": case, "pl": pl, "frames": fr, "k": 0}
        if kind == "filter":  # the frame up to its resolve is done: the case is the probe stage
            for f in fr:
                v = f["cam"].view(f["index"])
                pl.spawn(f["gbuf"], v)
                pl.update(f["rec"], v)
                pl.resolve(f["index"])
        else:
            run(s)
        return s
    if kind == "batch":
        bp = BatchPipeline([(w, h, n) for _, w, h, n in _batch_views(case)], 64)
        s = {"case": case, "bp": bp, "frames": _batch_frames(case, seed), "k": 0}
        run(s)
        return s
    if kind == "temporal":
        g = _gen(seed)
        sc = _scene("boxes", g)
        w, h, u = case["width"], case["height"], case["upscale"]
        cams = [_Cam(sc, f, w, h) for f in (0, 1)]
        # the camera sways between two positions: each frame's motion vectors lead to the other; the
        # first frame run after the history traces from that frame's own probe pixels
        fr = [_frame(sc, f, w, h, case["rpp"], g, u, 2 + f, cams[1 - f]) for f in (0, 1)]
        kw = {"tiles": True, "min_samples": 16} if case["tiles"] else {}
        tp = TemporalPipeline(w, h, case["rpp"], case["log2_slots"], upscale=u, filtered=case["filtered"], **kw)
        s = {"case": case, "tp": tp, "frames": fr, "k": 0}
        for _ in range(2):
            run(s)
        return s
    if kind == "cache":
        fr = _cache_frames(case, seed)
        n = case["n"]
        h = gi.gi_cache_create(case["log2_slots"], key_dir=case["key_dir"], resolved_format=int(case["f16"]),
                               first_touch=case["first_touch"], tiles=case["tiles"], merge=case["merge"])
        s = {"case": case, "cache": _Handle(gi.gi_cache_destroy, h), "frames": fr, "k": 0,
             "slots": torch.empty(n, dtype=torch.int32, device=DEV), "by_slot": torch.empty(n, 4, device=DEV),
             "by_point": torch.empty(n, 4, device=DEV)}
        run(s)
        return s
    if kind in ("train", "far"):
        small = dict(case, scene="cornell" if kind == "train" else "boxes", rpp=64)
        fr = _two(small, seed)
        n = fr[0]["rec"].shape[1]
        box = CORNELL_AABB if kind == "train" else ((-0.2,) * 3, tuple(x + 0.2 for x in ROOM))
        steps = case.get("steps", 4)
        cfg = gi.make_nrc_config(*box, log2_table=case["log2_table"], batch=case.get("batch", 65536), train_steps=steps,
                                 max_records=n, max_queries=min(n, gi.GI_NRC_MAX_BATCH), trust=1e30,
                                 lr=2e-2 if kind == "train" else 1e-30, seed=seed + 1)
        nrc = _Handle(gi.gi_nrc_destroy, gi.gi_nrc_create(cfg))
        pl = Pipeline(case["width"], case["height"], 64, case.get("log2_slots", 20))
        for f in fr:
            v = f["cam"].view(f["index"])
            pl.spawn(f["gbuf"], v)
            pl.update(f["rec"], v)
            pl.resolve(f["index"])
        hits = [gi.hits_from_planes(f["rec"], n) for f in fr]
        s = {"case": case, "pl": pl, "nrc": nrc, "frames": fr, "hits": hits, "k": 0, "n": n}
        if kind == "train":
            m = min(n, 65536)
            take = torch.randint(0, n, (m,), generator=_gen(seed + 3), device=DEV)
            s["points"] = gi.make_points(fr[1]["rec"][0:3, take].contiguous(), fr[1]["rec"][3:6, take].contiguous(), m)
            s["rad"] = torch.empty(m, 4, device=DEV)
            for k in range(4):  # the optimiser's moments have a history
                gi.gi_nrc_train_frame(nrc.h, pl.cache, hits[1], pl.slot_ids, k)
            s["k"] = 4
        else:  # an Adam step too small to move anything gives the network its trust; then a routed history
            gi.gi_nrc_train_frame(nrc.h, pl.cache, hits[1], pl.slot_ids, 0)
            gi.gi_cache_route_far(pl.cache, nrc.h, 2)
            s["k"] = 2
        return s
    prm, pos, nrm = _infer_inputs(case, seed)
    cfg = gi.make_nrc_config(*CORNELL_AABB, log2_table=case["log2_table"], max_records=128, max_queries=128)
    nrc = _Handle(gi.gi_nrc_destroy, gi.gi_nrc_create(cfg))
    gi.gi_nrc_set_params(nrc.h, *[p.cpu().numpy() for p in prm])
    return {"case": case, "nrc": nrc, "points": gi.make_points(pos, nrm, case["n"]), "rad": torch.empty(case["n"], 4, device=DEV)}


class _Handle:
    """A C-ABI handle freed with its state."""

    def __init__(self, free, h):
        self.free, self.h = free, h

    def __del__(self):
        try:
            self.free(self.h)
        except Exception:
            pass


def run(s):
    kind = s["case"]["kind"]
    if kind == "infer":
        gi.gi_nrc_infer(s["nrc"].h, s["points"], s["rad"])
        return s["rad"]
    if kind == "filter":
        f, pl = s["frames"][1], s["pl"]
        pl.integrate_filtered(f["rec"], f["cam"].view(1))
        return {"atlas": pl.atlas, "sh": pl.probes.sh}
    k = s["k"]
    s["k"] = k + 1
    if kind == "batch":
        bp, fr = s["bp"], [v[k % 2] for v in s["frames"]]
        bp.frame([f["gbuf"] for f in fr], [f["rec"] for f in fr], [f["cam"].view(f["index"]) for f in fr],
                 use_graph=s["case"]["graph"], resolve_frame=k)
        return [{"irr": st["irr"], "sh": st["probes"].sh, "mask": st["probes"].mask} for st in bp.views]
    f = s["frames"][k % 2]
    if kind == "frame":
        pl, v = s["pl"], f["cam"].view(f["index"])
        pl.spawn(f["gbuf"], v)
        pl.update(f["rec"], v)
        pl.resolve(k)
        pl.integrate()
        pl.interpolate(f["gbuf"], v)
        return {"irr": pl.irr, "sh": pl.probes.sh, "mask": pl.probes.mask}
    if kind == "temporal":
        tp = s["tp"]
        tp.frame(f["gbuf"], f["rec"], f["motion"], f["cam"].view(k))
        return {"irr": tp.irr, "sh": tp.probes.sh, "mask": tp.probes.mask, "atlas": tp.atlas, "src": tp.src}
    if kind == "cache":
        n, v, h = s["case"]["n"], f["cam"].view(f["index"]), s["cache"].h
        hits = gi.hits_from_planes(f["rec"], n)
        gi.gi_cache_update(h, hits, v, s["slots"])
        gi.gi_cache_resolve(h, k)
        gi.gi_cache_query(h, s["by_slot"], n, slot_ids=s["slots"], env=(0.1, 0.2, 0.3))
        other = s["frames"][(k + 1) % 2]
        gi.gi_cache_query(h, s["by_point"], n, points=gi.hits_from_planes(other["rec"], n),
                          view=other["cam"].view(other["index"]))
        return {"by_slot": s["by_slot"], "by_point": s["by_point"]}
    pl = s["pl"]
    if kind == "train":
        gi.gi_nrc_train_frame(s["nrc"].h, pl.cache, s["hits"][1], pl.slot_ids, k)
        # what the step leaves: the network's answer at points of the frame (through table and weights) and its
        # weights, which a user reads through the C ABI
        gi.gi_nrc_infer(s["nrc"].h, s["points"], s["rad"])
        w = [np.empty(x, np.float32) for x in ((64, 32), (64, 64), (3, 64))]
        gi.check(gi.lib().gi_nrc_get_params(s["nrc"].h, None, *[x.ctypes.data for x in w]), "gi_nrc_get_params")
        return {"rad": s["rad"], "weights": w}
    v = f["cam"].view(f["index"])
    pl.spawn(f["gbuf"], v)
    pl.update(f["rec"], v)
    pl.resolve(k)
    gi.gi_nrc_query_frame(s["nrc"].h, pl.cache, s["hits"][k % 2], pl.slot_ids, v)
    gi.gi_probes_integrate_nrc(pl.cache, s["nrc"].h, pl.probes.struct, pl.slot_ids, 64)
    return {"sh": pl.probes.sh, "mask": pl.probes.mask}


# ---------------------------------------------------------------------------------------- work

def _frame_work(w, h, rpp, upscale=1, f16=False, interpolate=True):
    """Records, slot ids and touched cells (about 0.4 per record: accumulate, blend, store), radiance per ray,
    probes, and per pixel the G-buffer and the irradiance."""
    st = 8 * upscale
    n = -(-w // st) * -(-h // st) * rpp
    probes = -(-w // 8) * -(-h // 8)
    cell = 32 + 2 * (8 if f16 else 16)
    return n, probes, 40 * n + 4 * n + 0.4 * n * cell + 16 * probes + 112 * probes + 36 * probes + (32 * w * h if interpolate else 0)


def work(case):
    kind = case["kind"]
    if kind == "infer":
        return {"bytes": case["n"] * (24 + 16 + 16 * 8 * 4.0), "flops": case["n"] * 2.0 * (32 * 64 + 64 * 64 + 64 * 3)}
    if kind == "train":
        b, m = case["batch"], min(65536, -(-case["width"] // 8) * -(-case["height"] // 8) * 64)
        touched = 0.5 * b * 128  # distinct table entries of a step: parameters and moments read and written
        return {"bytes": b * (28 + 20 + 128 * 4) + touched * (8 + 48 + 4) + m * (24 + 16 + 512.0),
                "flops": (3 * b + m) * 2.0 * (32 * 64 + 64 * 64 + 64 * 3)}
    if kind == "cache":
        n = case["n"]
        return {"bytes": n * (40 + 4 + 4 + 16 + 28 + 16) + 0.4 * n * (32 + 2 * (8 if case["f16"] else 16)), "flops": n * 60.0}
    if kind == "batch":
        return {"bytes": sum(_frame_work(w, h, 64)[2] for _, w, h, _ in _batch_views(case)),
                "flops": sum(w * h * 100.0 + w * h * 60 for _, w, h, _ in _batch_views(case))}
    w, h = case["width"], case["height"]
    n, probes, b = _frame_work(w, h, case.get("rpp", 64), case.get("upscale", 1), case.get("f16", False), kind not in ("far", "filter"))
    fl = n * 120.0 + (w * h * 100.0 if kind not in ("far", "filter") else 0)
    if kind == "filter":
        return {"bytes": n * (4 + 4 + 16) + probes * (32 + 112 + 3 * 2048.0), "flops": probes * 64 * 2 * 6 * 40.0}
    if kind == "temporal":
        atlas = probes * 1024.0
        b += 24 * w * h + 3 * atlas + (4 * atlas if case["filtered"] else 0)
        fl += probes * 64 * 2 * 6 * 40.0 if case["filtered"] else 0
    if kind == "far":
        far = 0.15 * n
        b += far * (24 + 512 + 16)
        fl += far * 2.0 * (32 * 64 + 64 * 64 + 64 * 3)
    return {"bytes": float(b), "flops": float(fl)}


# ---------------------------------------------------------------------------------------- exact values

def _keys(rec, cam, key_dir):
    """Cell of each record (the descriptor's float32 operations, one rounding each); -1 where it is no hit."""
    m = max(1 / cam.height, cam.height / cam.width ** 2)
    s0 = float(np.float32(CELL))
    d0 = s0 / math.tan(FOV * 8 * m)
    p, ln = rec[0:3], rec[9]
    q = p - torch.tensor(cam.pos, device=DEV)[:, None]
    q = q * q
    d2 = (q[0] + q[1]) + q[2]
    lod = torch.zeros_like(ln, dtype=torch.int64)
    for k in range(1, LODS):
        lod += d2 >= float(np.float32((d0 * 2.0 ** k) ** 2))
    inv0 = float(np.float32(1 / s0))
    inv = torch.tensor([inv0 * 0.5 ** k for k in range(4)], device=DEV)[lod]
    side = torch.tensor([s0 * 2.0 ** k for k in range(4)], device=DEV)[lod]
    c = torch.floor(p * inv).long() & ((1 << 19) - 1)
    src = rec[10:13].neg() if key_dir else rec[3:6]
    a = src.abs()
    axis = torch.where((a[0] >= a[1]) & (a[0] >= a[2]), 0, torch.where(a[1] >= a[2], 1, 2))
    code = 2 * axis + torch.signbit(src.gather(0, axis[None])[0]).long()
    key = (lod << 61) | ((ln < side).long() << 60) | (code << 57) | (c[0] << 38) | (c[1] << 19) | c[2]
    hit = torch.isfinite(ln) & (ln >= 0) & torch.isfinite(p).all(0)
    return torch.where(hit, key, -torch.ones_like(key))


def _cells(frames, key_dir):
    """Cell values after the frames were resolved in order: sorted keys, values (cells, 3), live cells."""
    ks = [_keys(f["rec"], f["cam"], key_dir) for f in frames]
    uniq = torch.unique(torch.cat(ks))
    uniq = uniq[uniq >= 0]
    val = torch.zeros(uniq.numel(), 3, dtype=torch.float64, device=DEV)
    old = torch.zeros(uniq.numel(), dtype=torch.bool, device=DEV)
    al = float(np.float32(ALPHA))
    for k, f in zip(ks, frames):
        h = k >= 0
        i = torch.searchsorted(uniq, k[h])
        cnt = torch.zeros_like(old, dtype=torch.float64).index_add_(0, i, torch.ones_like(i, dtype=torch.float64))
        mean = torch.zeros_like(val).index_add_(0, i, f["rec"][6:9, h].T.double()) / cnt.clamp(min=1)[:, None]
        new = torch.where(old[:, None], val + al * (mean - val), mean)
        val = torch.where((cnt > 0)[:, None], new, val)
        old |= cnt > 0
    return uniq, val


def _answers(uniq, val, key):
    i = torch.searchsorted(uniq, key.clamp(min=0)).clamp(max=max(uniq.numel() - 1, 0))
    found = (key >= 0) & (uniq[i] == key)
    return torch.where(found[:, None], val[i], torch.zeros((), dtype=torch.float64, device=DEV)), found


_MOMENTS = []


def _moments():
    """Per hemi-octahedral cell the solid angle, first and second moment of the direction, by Gauss-Legendre
    quadrature on the four triangles that the cell's diagonals cut (the map's creases run along them)."""
    if not _MOMENTS:
        x, wx = np.polynomial.legendre.leggauss(24)
        s, t = np.meshgrid((x + 1) / 2, (x + 1) / 2, indexing="ij")
        wt = np.outer(wx / 2, wx / 2)
        out = np.zeros((64, 13))
        for c in range(64):
            u0, v0 = -1 + (c % 8) / 4, -1 + (c // 8) / 4
            corner = [np.array(q) for q in ((u0, v0), (u0 + 0.25, v0), (u0 + 0.25, v0 + 0.25), (u0, v0 + 0.25))]
            mid = sum(corner) / 4
            for k in range(4):
                b, e = corner[k] - mid, corner[(k + 1) % 4] - mid
                uv = mid + s[..., None] * ((1 - t)[..., None] * b + t[..., None] * e)
                X, Y = (uv[..., 0] + uv[..., 1]) / 2, (uv[..., 0] - uv[..., 1]) / 2
                p = np.stack((X, Y, 1 - abs(X) - abs(Y)), -1)
                r = np.linalg.norm(p, axis=-1)
                dw = wt * s * abs(b[0] * e[1] - b[1] * e[0]) * 0.5 / r ** 3
                d = p / r[..., None]
                out[c, 0] += dw.sum()
                out[c, 1:4] += np.einsum("ij,ija->a", dw, d)
                out[c, 4:] += np.einsum("ij,ija,ijb->ab", dw, d, d).reshape(9)
        _MOMENTS.append(torch.tensor(out, device=DEV))
    return _MOMENTS[0]


def _exact_view(frames, rpp, key_dir):
    """Irradiance image, SH and no mask of frames[-1] after the earlier frames' history, in 64 bits."""
    f = frames[-1]
    cam, gb, rec = f["cam"], f["gbuf"], f["rec"]
    w, h = cam.width, cam.height
    uniq, val = _cells(frames, key_dir)
    rad, has = _answers(uniq, val, _keys(rec, cam, key_dir))
    has = has | (rec[9] == math.inf)  # a ray that left the scene brings the environment: black
    tw, th = -(-w // 8), -(-h // 8)
    P = tw * th
    rad, has = rad.reshape(P, rpp // 64, 64, 3), has.reshape(P, rpp // 64, 64, 1).double()
    cnt = has.sum(1)
    L = (rad * has).sum(1) / cnt.clamp(min=1)
    pop = (cnt > 0).double()
    back = L.sum(1, keepdim=True) / pop.sum(1, keepdim=True).clamp(min=1)
    L = torch.where(cnt > 0, L, back)
    ty, tx = torch.meshgrid(torch.arange(th, device=DEV), torch.arange(tw, device=DEV), indexing="ij")
    px = (8 * tx + _halton(f["index"] + 1, 2, 8)).clamp(max=w - 1).reshape(-1)
    py = (8 * ty + _halton(f["index"] + 1, 3, 8)).clamp(max=h - 1).reshape(-1)
    nd = gb[py, px].double()
    valid = torch.isfinite(nd[:, 3])
    n = torch.where(valid[:, None], nd[:, :3], torch.tensor((0.0, 0.0, 1.0), device=DEV).double())
    M = torch.einsum("cm,pcx->pmx", _moments(), L)
    t, b = _frame_basis(n)
    R = torch.stack((t, b, n), -1)
    S0, S1 = M[:, 0], R @ M[:, 1:4]
    S2 = torch.einsum("pia,pjb,pabx->pijx", R, R, M[:, 4:].reshape(P, 3, 3, 3))
    c1, c2 = math.sqrt(3 / (4 * math.pi)), math.sqrt(15 / (4 * math.pi))
    sh = torch.stack((S0 * math.sqrt(1 / (4 * math.pi)), c1 * S1[:, 1], c1 * S1[:, 2], c1 * S1[:, 0], c2 * S2[:, 0, 1],
                      c2 * S2[:, 1, 2], math.sqrt(5 / (16 * math.pi)) * (3 * S2[:, 2, 2] - S0), c2 * S2[:, 0, 2],
                      0.5 * c2 * (S2[:, 0, 0] - S2[:, 1, 1])), 1)
    sh = torch.where(valid[:, None, None], sh, torch.zeros((), dtype=torch.float64, device=DEV))
    pos = torch.tensor(cam.pos, device=DEV).double() + cam.rays(px, py, torch.float64) * torch.where(valid, nd[:, 3], torch.zeros((), device=DEV).double())[:, None]
    level = torch.where(valid, torch.arange(P, device=DEV), -torch.ones(P, dtype=torch.int64, device=DEV)).reshape(th, tw)
    mips = [level]
    while max(mips[-1].shape) > 1:
        m = mips[-1]
        H2, W2 = (m.shape[0] + 1) // 2, (m.shape[1] + 1) // 2
        pad = -torch.ones(2 * H2, 2 * W2, dtype=torch.int64, device=DEV)
        pad[:m.shape[0], :m.shape[1]] = m
        o = pad[0::2, 0::2]
        for c in (pad[0::2, 1::2], pad[1::2, 0::2], pad[1::2, 1::2]):
            o = torch.where(o < 0, c, o)
        mips.append(o)
    out = torch.empty(h, w, 4, dtype=torch.float64, device=DEV)
    shz = torch.cat((sh.reshape(P, 27), torch.zeros(P, 1, dtype=torch.float64, device=DEV)), 1)
    rows = max(8, (1 << 21) // w)
    for y0 in range(0, h, rows):
        ys, xs = torch.meshgrid(torch.arange(y0, min(h, y0 + rows), device=DEV), torch.arange(w, device=DEV), indexing="ij")
        nd = gb[y0:y0 + rows].double()
        sky = ~(torch.isfinite(nd[..., 3]) & (nd[..., 3] >= 0))
        dist = torch.where(sky, torch.ones_like(nd[..., 3]), nd[..., 3])
        nn = nd[..., :3]
        Pp = torch.tensor(cam.pos, device=DEV).double() + cam.rays(xs, ys, torch.float64) * dist[..., None]
        cs = math.tan(FOV * 8 * max(1 / h, h / w ** 2)) * dist
        bx, by = torch.div(xs - 4, 8, rounding_mode="floor"), torch.div(ys - 4, 8, rounding_mode="floor")
        fx, fy = (xs + 0.5 - 4) / 8 - bx, (ys + 0.5 - 4) / 8 - by
        x, y, z = nn.unbind(-1)
        A0, A1, A2 = math.pi, 2 * math.pi / 3, math.pi / 4
        Y = torch.stack((torch.full_like(x, A0 * math.sqrt(1 / (4 * math.pi))), A1 * c1 * y, A1 * c1 * z, A1 * c1 * x,
                         A2 * c2 * x * y, A2 * c2 * y * z, A2 * math.sqrt(5 / (16 * math.pi)) * (3 * z * z - 1),
                         A2 * c2 * x * z, A2 * 0.5 * c2 * (x * x - y * y)), -1)
        ws, es, er, nf = 0, 0, 0, 0
        for ox, oy in ((0, 0), (1, 0), (0, 1), (1, 1)):
            q = -torch.ones_like(xs)
            go, cx, cy = torch.ones_like(sky), bx, by
            for m in mips:
                X, Yy = cx + ox, cy + oy
                go = go & (X >= 0) & (Yy >= 0) & (X < m.shape[1]) & (Yy < m.shape[0])
                e = torch.where(go, m[Yy.clamp(0, m.shape[0] - 1), X.clamp(0, m.shape[1] - 1)], -torch.ones_like(xs))
                q = torch.where(e >= 0, e, q)
                go = go & (e < 0)
                cx, cy = cx >> 1, cy >> 1
            ok = (q >= 0) & ~sky
            qi = q.clamp(min=0)
            E = torch.einsum("yxk,yxkc->yxc", Y, sh[qi]) * ok[..., None]
            dot = (nn * n[qi]).sum(-1).clamp(min=0) ** 8
            wd = (1 - ((pos[qi] - Pp) * nn).sum(-1).abs() / cs).clamp(min=0)
            wt = (fx if ox else 1 - fx) * (fy if oy else 1 - fy) * dot * wd * ok
            ws, es, er, nf = ws + wt, es + wt[..., None] * E, er + E, nf + ok.long()
        good = ws > 0
        r = torch.where(good[..., None], es / torch.where(good, ws, torch.ones_like(ws))[..., None], er / nf.clamp(min=1)[..., None])
        flag = torch.where(sky, 3.0, torch.where(nf == 0, 2.0, torch.where(good, 0.0, 1.0)))
        r = torch.where(sky[..., None], torch.zeros((), dtype=torch.float64, device=DEV), r)
        out[y0:y0 + rows] = torch.cat((r, flag[..., None].double()), -1)
    return {"irr": out, "sh": shz, "mask": None}


def _exact_infer(case, seed):
    prm, pos, nrm = _infer_inputs(case, seed)
    table, w1, w2, w3 = (p.double() for p in prm)
    T = 1 << case["log2_table"]
    lo, hi = (torch.tensor(v, device=DEV) for v in CORNELL_AABB)
    inv = torch.tensor([np.float32(1 / (float(b) - float(a))) for a, b in zip(lo.tolist(), hi.tolist())], device=DEV)
    x = ((pos - lo[:, None]) * inv[:, None]).clamp(0, 1)
    a = nrm.abs()
    axis = torch.where((a[0] >= a[1]) & (a[0] >= a[2]), 0, torch.where(a[1] >= a[2], 1, 2))
    code = 2 * axis + torch.signbit(nrm.gather(0, axis[None])[0]).long()
    feats = []
    for l, R in enumerate(gi.default_resolutions()):
        s = x * float(R)
        i = torch.floor(s).long().clamp(max=R - 1)
        f = (s - i).double()
        V = R + 1
        e = 0
        for c in range(8):
            o = (c & 1, c >> 1 & 1, c >> 2 & 1)
            v = [i[k] + o[k] for k in range(3)]
            if 6 * V ** 3 <= T:
                idx = ((code * V + v[2]) * V + v[1]) * V + v[0]
            else:
                idx = (v[0] ^ (v[1] * 2654435761) ^ (v[2] * 805459861) ^ (code * 2246822519)) & (T - 1)
            wt = 1
            for k in range(3):
                wt = wt * (f[k] if o[k] else 1 - f[k])
            e = e + wt[:, None] * table[l][idx]
        feats.append(e)
    z = torch.cat(feats, 1)
    z = torch.relu(torch.relu(z @ w1.T) @ w2.T) @ w3.T
    return torch.cat((torch.relu(z), torch.ones_like(z[:, :1])), 1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "infer":
        return _exact_infer(case, seed)
    if kind == "frame":
        return _exact_view(_two(case, seed), case["rpp"], case["key_dir"])
    if kind == "batch":
        return [_exact_view(fr, 64, 0) for fr in _batch_frames(case, seed)]
    if kind == "cache" and not case["tiles"]:
        fr = _cache_frames(case, seed)
        uniq, val = _cells(fr, case["key_dir"])
        out = {}
        for name, f in (("by_slot", fr[1]), ("by_point", fr[0])):
            v, found = _answers(uniq, val, _keys(f["rec"], f["cam"], case["key_dir"]))
            v = torch.cat((v, found[:, None].double()), 1)
            if name == "by_slot":
                v[f["rec"][9] == math.inf] = torch.tensor((0.1, 0.2, 0.3, 1.0), device=DEV).double()
            out[name] = v
        return out
    # the tile cache's level rule, the temporal blends, the filter's decisions and the bfloat16 training and
    # query steps have no value of their own in 64 bits that is not this path again
    return None
