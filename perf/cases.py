"""Performance cases of the Flow Fields matching library: what its users have it do, through the public binding.

A case is a dict of plain values.  ``op`` names the call sequence, the rest are sizes and matching parameters:

* ``frames``     ``Matcher.match_frames`` on ``n`` image pairs (features and matching in one call);
* ``track``      features of one new frame, matched against a kept pyramid with two consistency checks, and the
                 3x3 sparsification of what they left (the whole filter of FlowFields++ Sec. 3.1);
* ``direction``  ``Matcher.match_pair``: one direction between two existing pyramids, with costs;
* ``noalloc``    ``ff_match_pair_noalloc``: the same for callers that must not allocate;
* ``features``   ``Matcher.features_batch`` on ``n`` frames (the descriptors themselves are the result);
* ``serve``      ``n`` requests of mixed sizes through the continuous-batching server, all arriving at once.

Every output is a whole number (flows, costs, masks, integer descriptors), so there is nothing to compare with in
64-bit floating point: results have to be equal.

Frames are made on the device from the seed alone, with the scene kinds of the package's synthetic pairs: a driving
scene (ground plane under forward motion, up to 250 px of flow, boxes), an animation (rotating, scaling, shifted
sprites, gain, noise) and translated rectangles over value noise.
"""
from __future__ import annotations

import json
import math
import os

import torch

from paper_1805_03517_gb300 import configs, ff

_TABLE = os.path.join(os.path.dirname(ff.__file__), "tuned.json")
_SIZES = [(w, h, kind) for w, h, kind in configs.SERVE_SIZES]


def _case(name, op, w, h, scene, **kw):
    c = {"name": name, "op": op, "w": w, "h": h, "scene": scene, "n": 1, "levels": 5, "iters": 6, "eps": 1, "cost": 0,
         "sub_scales": 0, "costs": False, "table": False, "mixed": False}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest pair the package is configured for: latency and launches count
        _case("pair_128x96", "frames", 128, 96, "rects", levels=3, iters=4),
        # one driving-size pair at a time, out of the box: an untuned context, as a new user has it
        _case("pair_1242x375", "frames", 1242, 375, "kitti"),
        # the same with the package's table of launch configurations, as a latency-critical loop sets it up
        _case("pair_1242x375_table", "frames", 1242, 375, "kitti", table=True),
        # one animation-size pair under the Census cost (the cost FlowFields++ takes there), costs wanted too
        _case("pair_1024x436_census", "frames", 1024, 436, "sintel", eps=7, cost=1, costs=True),
        # one full-HD pair: the largest single frames in everyday use
        _case("pair_1920x1080", "frames", 1920, 1080, "sintel", eps=7),
        # video: each new frame against a kept reference frame, with the whole filter (two checks, sparsification)
        _case("track_1242x375_filtered", "track", 1242, 375, "kitti"),
        # sub-scales and sub-sub-scales, the finer schedule of Sec. 3.1
        _case("pair_640x480_sub_scales", "frames", 640, 480, "rects", sub_scales=2),
        # one inverse field of an odd-sized pair between existing pyramids, with the paper's 12 iterations
        _case("direction_333x251", "direction", 333, 251, "rects", levels=4, iters=12, costs=True),
        # a real-time loop that must not allocate
        _case("noalloc_640x480", "noalloc", 640, 480, "rects", costs=True),
        # descriptors only: a program that extracts features of several frames for its own use
        _case("features_3x1920x1080", "features", 1920, 1080, "sintel", n=3),
        # offline processing: the 48-pair batch of mixed sizes, the largest call of the package's benchmark
        _case("batch48_mixed", "frames", 1242, 375, "kitti", n=48, mixed=True),
        # serving: sixteen requests of the served sizes that arrive together
        _case("serve_16_mixed", "serve", 1242, 375, "kitti", n=16, mixed=True),
    ]


def draw(rng):
    """One more case over the same ranges: sizes log-uniform in their pixels, any aspect from 1:1 to 4:1, odd ones."""
    op = rng.choice(["frames"] * 6 + ["track", "direction", "noalloc", "features", "serve"])
    px = math.exp(rng.uniform(math.log(96 * 72), math.log(1920 * 1080)))
    if op == "noalloc":
        px = min(px, 1.2e6)
    aspect = math.exp(rng.uniform(0.0, math.log(4.0)))
    w = max(64, int(math.sqrt(px * aspect)))
    h = max(48, int(px / w))
    levels = 3 if w * h < 30000 else rng.choice([4, 5]) if w * h < 400000 else 5
    iters = rng.choice([4, 6, 6, 12])
    most = max(1, min(48, int(80e6 / (w * h * iters))))
    n = 1
    if op in ("frames", "features") and rng.random() < 0.4:
        n = int(math.exp(rng.uniform(0.0, math.log(most if op == "frames" else min(most, 8)))))
    if op == "serve":
        n = rng.randint(2, min(16, max(2, most)))
    scene = rng.choice(["kitti", "sintel", "rects"])
    census = op in ("frames", "direction", "noalloc") and rng.random() < 0.25
    sub = rng.choice([1, 2]) if op == "frames" and n == 1 and w * h < 900000 and rng.random() < 0.2 else 0
    c = _case("", op, w, h, scene, n=n, levels=levels, iters=iters, eps=7 if scene == "sintel" else 1,
              cost=1 if census else 0, sub_scales=sub, costs=op in ("direction", "noalloc") or rng.random() < 0.3,
              mixed=op == "serve" and rng.random() < 0.5)
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------------------------
# inputs


class _Texture:
    """RGB value noise sampled at real coordinates (bilinear lattice of four octaves, stretched for contrast)."""

    def __init__(self, gen, dev, period, octaves=4):
        self.tab = torch.rand((octaves, 256 * 256, 3), generator=gen, device=dev)
        self.period, self.octaves = period, octaves

    def sample(self, x, y):
        out = 0.0
        for o in range(self.octaves):
            u, v = x / (self.period / 2 ** o), y / (self.period / 2 ** o)
            fu, fv = torch.floor(u), torch.floor(v)
            tu, tv = u - fu, v - fv
            tu, tv = (tu * tu * (3 - 2 * tu))[..., None], (tv * tv * (3 - 2 * tv))[..., None]
            iu, iv = fu.long() & 255, fv.long() & 255
            iu1, iv1 = (iu + 1) & 255, (iv + 1) & 255
            t = self.tab[o]
            a, b, c, d = t[iv * 256 + iu], t[iv * 256 + iu1], t[iv1 * 256 + iu], t[iv1 * 256 + iu1]
            out = out + 0.5 ** o * ((a * (1 - tu) + b * tu) * (1 - tv) + (c * (1 - tu) + d * tu) * tv)
        out = out / sum(0.5 ** o for o in range(self.octaves))
        return 20.0 + 215.0 * ((out - 0.5) * 2.2 + 0.5).clamp(0, 1)


def _numbers(gen, dev, n):
    """n numbers in [0, 1) on the host."""
    return torch.rand(n, generator=gen, device=dev).tolist()


def _u8(img):
    return img.round().clamp(0, 255).to(torch.uint8).contiguous()


def _kitti(gen, dev, w, h):
    r = _numbers(gen, dev, 40)
    f, cx, cy, cam = 0.58 * w, 0.5 * w + 20 * r[0] - 10, 0.42 * h, 1.65
    ground, sky = _Texture(gen, dev, 24.0), _Texture(gen, dev, 40.0)
    yb = (h - 1) - cy
    dz = f * cam / yb - f * cam / (yb + 250.0 * w / 1242)
    lateral = 0.3 * r[1] - 0.15
    ys, xs = torch.meshgrid(torch.arange(h, device=dev).float(), torch.arange(w, device=dev).float(), indexing="ij")
    below = ys > cy + 0.5
    z = f * cam / (ys - cy).clamp(min=0.6)
    imgs = []
    boxes = []
    for k in range(4):
        q = r[4 + 8 * k:12 + 8 * k]
        bw, bh = (0.06 + 0.1 * q[0]) * w, (0.12 + 0.18 * q[1]) * h
        bx, by = 0.05 * w + q[2] * (0.9 * w - bw), cy - 0.4 * bh + q[3] * (min(h - bh, cy + 0.5 * bh) - cy + 0.4 * bh)
        boxes.append((bx, by, bw, bh, 80 * q[4] - 40, 12 * q[5] - 6, _Texture(gen, dev, 10 + 10 * q[6])))
    for k in range(2):
        gx, gz = (xs - cx) * z / f + lateral * k, z + dz * k
        img = torch.where(below[..., None], ground.sample(gx * 30, gz * 30), sky.sample(xs, ys))
        for bx, by, bw, bh, mx, my, tex in boxes:
            x0, y0 = bx + k * mx, by + k * my
            hit = (xs >= x0) & (xs < x0 + bw) & (ys >= y0) & (ys < y0 + bh)
            img = torch.where(hit[..., None], tex.sample(xs - x0, ys - y0), img)
        imgs.append(img)
    imgs[1] = imgs[1] + torch.randn(imgs[1].shape, generator=gen, device=dev)
    return _u8(imgs[0]), _u8(imgs[1])


def _sintel(gen, dev, w, h):
    r = _numbers(gen, dev, 80)
    ys, xs = torch.meshgrid(torch.arange(h, device=dev).float(), torch.arange(w, device=dev).float(), indexing="ij")
    layers = []
    for k in range(6):
        q = r[12 * k:12 * k + 12]
        if k == 0:  # the backdrop covers the frame
            hw, hh, c, t = 0.8 * w, 0.8 * h, (0.5 * w, 0.5 * h), (80 * q[0] - 40, 80 * q[1] - 40)
        else:
            hw, hh, c = (0.08 + 0.17 * q[2]) * w, (0.1 + 0.25 * q[3]) * h, (q[4] * w, q[5] * h)
            t = (300 * q[0] * math.cos(2 * math.pi * q[1]), 300 * q[0] * math.sin(2 * math.pi * q[1]))
        a, da = math.radians(40 * q[6] - 20), math.radians(20 * q[7] - 10)
        s, ds = 0.9 + 0.2 * q[8], 0.9 + 0.2 * q[9]
        layers.append((hw, hh, (c, a, s), ((c[0] + t[0], c[1] + t[1]), a + da, s * ds), k > 0 and q[10] < 0.5,
                       _Texture(gen, dev, 12 + 18 * q[11])))
    imgs = []
    for k in range(2):
        img = torch.full((h, w, 3), 128.0, device=dev)
        for L in layers:
            (cx, cy), a, s = L[2 + k]
            dx, dy = xs - cx, ys - cy
            lx, ly = (math.cos(a) * dx + math.sin(a) * dy) / s, (-math.sin(a) * dx + math.cos(a) * dy) / s
            hit = (lx / L[0]) ** 2 + (ly / L[1]) ** 2 <= 1 if L[4] else (lx.abs() <= L[0]) & (ly.abs() <= L[1])
            img = torch.where(hit[..., None], L[5].sample(lx, ly), img)
        imgs.append(img)
    imgs[1] = imgs[1] * (0.95 + 0.1 * r[72]) + 3 * torch.randn(imgs[1].shape, generator=gen, device=dev)
    return _u8(imgs[0]), _u8(imgs[1])


def _rects(gen, dev, w, h):
    r = _numbers(gen, dev, 16)
    ys, xs = torch.meshgrid(torch.arange(h, device=dev).float(), torch.arange(w, device=dev).float(), indexing="ij")
    a = _u8(_Texture(gen, dev, 32.0).sample(xs, ys))
    b = a.clone()
    for k in range(2):
        q = r[8 * k:8 * k + 8]
        rw, rh = int(w / 6 + q[0] * w / 6), int(h / 6 + q[1] * h / 6)
        x0, y0 = int(q[2] * (w - rw)), int(q[3] * (h - rh))
        dx, dy = int(25 * q[4]) - 12, int(25 * q[5]) - 12
        xa, xb, ya, yb = max(0, x0 + dx), min(w, x0 + rw + dx), max(0, y0 + dy), min(h, y0 + rh + dy)
        b[ya:yb, xa:xb] = a[ya - dy:yb - dy, xa - dx:xb - dx]
    return a, _u8(b.float() + 2 * torch.randn(b.shape, generator=gen, device=dev))


_SCENES = {"kitti": _kitti, "sintel": _sintel, "rects": _rects}


def _sizes(case):
    """(w, h, scene) of each of the case's pairs."""
    if not case["mixed"]:
        return [(case["w"], case["h"], case["scene"])] * case["n"]
    if case["op"] == "serve":
        return [_SIZES[i % len(_SIZES)] for i in range(case["n"])]
    three = [(1242, 375, "kitti"), (1024, 436, "sintel"), (640, 480, "rects")]
    return [three[i * 3 // case["n"]] for i in range(case["n"])]


# ------------------------------------------------------------------------------------------------------------
# the calls


def _outputs(sizes, dev, costs, second=False):
    """Output buffers of many pairs: one allocation per kind, and each pair's views of them."""
    total = sum(w * h for w, h, _ in sizes)
    flat = {"flow_fwd": torch.zeros((total, 2), dtype=torch.int16, device=dev),
            "flow_bwd": torch.zeros((total, 2), dtype=torch.int16, device=dev),
            "mask": torch.zeros((total,), dtype=torch.uint8, device=dev)}
    if costs:
        flat["cost_fwd"] = torch.zeros((total,), dtype=torch.int32, device=dev)
        flat["cost_bwd"] = torch.zeros((total,), dtype=torch.int32, device=dev)
    if second:
        flat["flow_bwd2"] = torch.zeros((total, 2), dtype=torch.int16, device=dev)
    outs, o = [], 0
    for w, h, _ in sizes:
        outs.append({k: v[o:o + w * h].view((h, w, 2) if v.dim() == 2 else (h, w)) for k, v in flat.items()})
        o += w * h
    return flat, outs


_stream = []


def _shared_stream():
    """One stream for every context of the no-allocation call: its calls share one scratch array and have to be
    serialised by the caller."""
    if not _stream:
        _stream.append(torch.cuda.Stream(device=0))
    return _stream[0]


def prepare(case, seed):
    dev = torch.device("cuda", 0)
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed * 7919 + 17)
    prm = configs.MatchParams(n_scales=case["levels"], iters=case["iters"], eps=case["eps"], cost=case["cost"],
                              sub_scales=case["sub_scales"])
    M = ff.Matcher(prm, 0, _shared_stream() if case["op"] == "noalloc" else None)
    if case["table"]:
        with open(_TABLE) as f:
            for level, cfg in enumerate(json.load(f)["kitti_1242x375"]):
                ff.ff_set_tuning(M.ctx, level, cfg)
    sizes = _sizes(case)
    st = {"case": case, "M": M, "pairs": [_SCENES[s](gen, dev, w, h) for w, h, s in sizes]}
    op = case["op"]
    if op in ("frames", "track", "serve"):
        st["flat"], st["outs"] = _outputs(sizes, dev, case["costs"], op == "track")
    torch.cuda.synchronize()
    a, b = st["pairs"][0]
    if op == "track":
        st["ref"] = M.features(a)
    elif op in ("direction", "noalloc"):
        st["a"], st["b"] = M.features(a), M.features(b)
        st["flow"] = torch.zeros((case["h"], case["w"], 2), dtype=torch.int16, device=dev)
        st["cost"] = torch.zeros((case["h"], case["w"]), dtype=torch.int32, device=dev)
    elif op == "features":
        st["frames"] = [p[0] for p in st["pairs"]]
        st["pyrs"] = []
    elif op == "serve":
        st["srv"] = ff.Server(M, 60 << 30, 256)
        st["next"] = 0
    M.sync()
    torch.cuda.synchronize()
    return st


def run(st):
    case, M = st["case"], st["M"]
    op = case["op"]
    if op == "frames":
        M.match_frames(st["pairs"], st["outs"], with_cost=case["costs"])
        return st["flat"]
    if op == "track":
        new = M.features(st["pairs"][0][1])
        out = M.match_batch([(st["ref"], new)], st["outs"])[0]
        sparse = M.sparsify(out["flow_fwd"], out["flow_bwd"], case["eps"], 7, out["mask"])
        M.release(new)
        return {**st["flat"], "sparse": sparse}
    if op == "direction":
        flow, cost = M.match_pair(st["a"], st["b"], 1)
        return {"flow": flow, "cost": cost}
    if op == "noalloc":
        ff.ff_match_pair_noalloc(M.ctx, st["a"].handle, st["b"].handle, 0, st["flow"].data_ptr(), st["cost"].data_ptr())
        return {"flow": st["flow"], "cost": st["cost"]}
    if op == "features":
        for p in st["pyrs"]:
            M.release(p)
        st["pyrs"] = M.features_batch(st["frames"])
        got = []
        for p in st["pyrs"]:  # the descriptors in place, as a consumer on the device reads them
            for s in range(case["levels"]):
                w, h = ff.ff_pyr_level_dims(p.handle, s)
                view = ff._DevView(ff.ff_pyr_features(p.handle, s), w * h * 96)
                view.owner = M  # the pyramid's memory lives as long as its context; the tensor keeps the view
                got.append(torch.as_tensor(view, device=M.device).view(torch.int16).view(h, w, 48))
        return got
    srv, first = st["srv"], st["next"]
    st["next"] += case["n"]
    for i, ((a, b), out) in enumerate(zip(st["pairs"], st["outs"])):
        srv.submit(first + i, a, b, out)
    left = case["n"]
    while left:
        active, queued = srv.step()
        left -= len(srv.poll(wait=active == 0 and queued == 0))
    return st["flat"]


def work(case):
    """Bytes: the frames once, the outputs once.  Operations: the descriptors (a separable 8x8 -> 4x4 transform per
    channel and frame), the exhaustive initial matches (64 products per pixel pair of the coarsest level), and per
    pixel, iteration and direction the distances to its three random candidates (48 differences and sums each; the
    neighbours' candidates need not be scored again while nothing around a pixel changes)."""
    nbytes = ops = 0
    L, T, op = case["levels"], case["iters"], case["op"]
    dirs = 1 if op in ("direction", "noalloc") else 0 if op == "features" else 3 if op == "track" else 2
    coef = 6 if case["cost"] else 48
    for w, h, _ in _sizes(case):
        px = w * h
        level_px = [max(1, w >> s) * max(1, h >> s) for s in range(L)]
        if op == "features":
            nbytes += px * 3 + sum(level_px) * 96
            ops += sum(level_px) * 3 * 2 * (8 * 4 + 4 * 4) * 2
            continue
        if op in ("direction", "noalloc"):  # the descriptors exist: read once each
            nbytes += 2 * sum(level_px) * (32 if case["cost"] else 96)
        else:
            nbytes += 2 * px * 3
            ops += 2 * sum(level_px) * 3 * 2 * (8 * 4 + 4 * 4) * 2
        nbytes += dirs * px * (8 if case["costs"] else 4) + (0 if op in ("direction", "noalloc") else px)
        ops += dirs * (2 * 64 * level_px[-1] ** 2 + sum(level_px) * T * 3 * 2 * coef)
        if op == "track":
            nbytes += px
    return {"bytes": nbytes, "flops": ops}
