"""The work whose time counts: what programs ask of this library, call by call.

A case is a dict of plain values.  ``kind`` names the path, ``layout`` seeds the
geometry (which rectangles the sources cover), so that the bytes of a pass
follow from the case alone; the pixel values follow from the seed given to
``prepare``.  Everything runs on the current CUDA device and stream.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1902_08755_gb300 as ec

# ------------------------------------------------------------------- cases


def listed():
    return [
        # Smallest merge: four uncropped 640x480 partial frames, with the winner
        # plane an interactive viewer picks from.  Launch and host time count.
        dict(name="merge_vga", kind="merge", n=4, w=640, h=480, cover=0.4, cropped=False, align=4, winner=True,
             layout=1),
        # An ordinary sort-last frame: 16 ROI-cropped 1080p sources are
        # compressed (colour swizzled), decompressed and merged.
        dict(name="frame_hd", kind="frame", n=16, w=1920, h=1080, cover=0.3, cropped=True, align=4, layout=2),
        # A display wall's frame: the same over 16 sources of 7680x4320.
        dict(name="frame_8k", kind="frame", n=16, w=7680, h=4320, cover=0.25, cropped=True, align=4, layout=5),
        # Smoothly shaded geometry: nearly every pixel's colour and depth differ
        # from the neighbour's, so runs are short (compress and decompress).
        dict(name="shaded_hd", kind="shaded", n=8, w=1920, h=1080, cover=0.3, align=4, layout=6),
        # Slow links: colour through the lossy YUV codec and the RLE, and back;
        # crops of odd width, so rows start at any element.
        dict(name="yuv_hd", kind="yuv", n=8, w=1917, h=1079, cover=0.3, align=1, layout=7),
        # Parallel volume rendering: 32 slabs of 2048x2048, FP32, blended in
        # view order, with the remaining transmittance for the background.
        dict(name="over_f32", kind="over", n=32, w=2048, h=2048, half=False, cropped=False, back=True, amax=0.3,
             layout=3),
        # Inverse rendering, small: forward and backward over 12 FP32 layers of
        # a ragged 333x257 crop, each layer covering a part of it.
        dict(name="train_small_f32", kind="train", n=12, w=333, h=257, half=False, cropped=True, back=False, amax=0.3,
             layout=8),
        # Inverse rendering, deep: 128 FP16 slices of 1920x1080, gradients FP16.
        dict(name="train_deep_f16", kind="train", n=128, w=1920, h=1080, half=True, cropped=False, back=False,
             amax=0.1, layout=9),
        # A cluster's exchange: binary swap of 16 1080p sources with RLE
        # transfers, one captured graph per frame.
        dict(name="swap_hd", kind="swap", n=16, w=1920, h=1080, cover=0.3, algorithm="binary_swap", layout=2),
        # Many views at once: 128 uneven composites (sides 16 to 1024, 2 to 64
        # layers, depth and alpha in turn) in one planned launch.
        dict(name="batch_uneven", kind="batch", n=128, side=1024, layers=64, layout=4),
        # Sort-first display: a 3840x2160 frame put together from 64 tiles whose
        # borders follow the load, at any pixel.
        dict(name="sortfirst_4k", kind="tiles", nx=8, ny=8, w=3840, h=2160, half=False, layout=10),
        # Regions of interest found on the device: 16 uncropped 1080p sources.
        dict(name="roi_hd", kind="roi", n=16, w=1920, h=1080, cover=0.3, tile=64, layout=2),
    ]


# (width, height) range of a frame: a thumbnail to a display wall
_SMALL, _LARGE = 96, 7680
_MOST_BYTES = 4.0e9                               # a drawn case moves no more than this
_MOST_STORED = 2.0e9                              # and its sources hold no more than this


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above: a frame of 96 to 7680 columns in any
    aspect of screens, 2 to 64 sources (128 layers), odd sizes as often as even."""
    while True:
        kind = rng.choice(["merge", "frame", "frame", "shaded", "yuv", "over", "train", "swap", "batch", "tiles", "roi"])
        w = _log_int(rng, _SMALL, _LARGE)
        h = max(48, int(w * rng.uniform(0.45, 1.1)))
        if rng.random() < 0.5:
            w = (w + 3) // 4 * 4                  # a multiple of four, as screens have
        c = dict(kind=kind, n=_log_int(rng, 2, 64), w=w, h=h, layout=rng.randrange(1 << 30))
        if kind in ("merge", "frame", "shaded", "yuv", "swap", "roi"):
            c.update(cover=round(rng.uniform(0.15, 0.45), 2))
        if kind in ("merge", "frame"):
            c.update(cropped=rng.random() < 0.75)
        if kind in ("merge", "frame", "shaded", "yuv"):
            c.update(align=rng.choice([1, 4, 4, 4]))
        if kind == "merge":
            c.update(winner=rng.random() < 0.5)
        if kind in ("shaded", "yuv"):
            c.update(n=_log_int(rng, 1, 16))
        if kind in ("over", "train"):
            c.update(n=_log_int(rng, 2, 128), half=rng.random() < 0.5, cropped=rng.random() < 0.4,
                     back=rng.random() < 0.5)
            c.update(amax=0.3 if c["n"] <= 64 else 0.1)
        if kind == "swap":
            c.update(n=_log_int(rng, 2, 16),
                     algorithm=rng.choice(["binary_swap", "binary_swap", "direct_send", "two_three_swap", "stream"]))
        if kind == "batch":
            c = dict(kind=kind, n=_log_int(rng, 8, 128), side=_log_int(rng, 128, 1024), layers=rng.randint(4, 64),
                     layout=c["layout"])
        if kind == "tiles":
            c = dict(kind=kind, nx=rng.randint(1, 8), ny=rng.randint(1, 8), w=w, h=h, half=rng.random() < 0.3,
                     layout=c["layout"])
        if kind == "roi":
            c.update(tile=rng.choice([8, 16, 32, 64]))
        stored = 16.0 * c.get("n", 1) * w * h if kind not in ("batch", "tiles") else 0.0
        if kind in ("merge", "frame") and c["cropped"]:
            stored *= 2 * c["cover"]
        if stored <= 4 * _MOST_STORED and work(c)["bytes"] <= _MOST_BYTES:
            return c


# ---------------------------------------------------------------- geometry


def _layout(case, i):
    return np.random.Generator(np.random.PCG64([case["layout"], i]))


def _boxes(case, i):
    """Source i's rectangles (x, y, w, h): compact geometry (its parts lie in a
    random sub-rectangle about twice the covered area), or spread over the
    frame where the source is not cropped; at most 64 parts."""
    W, H, cover = case["w"], case["h"], case["cover"]
    r = _layout(case, i)
    if case.get("cropped", True):
        area = min(1.0, 2.0 * cover) * W * H
        aspect = math.exp(r.uniform(math.log(0.75), math.log(4.0 / 3.0)))
        rw = int(min(W, max(8, round(math.sqrt(area * aspect)))))
        rh = int(min(H, max(8, round(area / rw))))
        rx, ry, part = int(r.integers(0, W - rw + 1)), int(r.integers(0, H - rh + 1)), 0.5
    else:
        rx, ry, rw, rh, part = 0, 0, W, H, cover
    # a part covers about 0.0244 of the region; n of them 1 - (1 - 0.0244)^n
    n = int(min(64, max(1, round(math.log(1.0 - part) / math.log(1.0 - 0.0244)))))
    out = []
    for _ in range(n):
        bw = int(max(1, min(rw, round(r.uniform(1 / 16, 1 / 4) * rw))))
        bh = int(max(1, min(rh, round(r.uniform(1 / 16, 1 / 4) * rh))))
        out.append((rx + int(r.integers(0, rw - bw + 1)), ry + int(r.integers(0, rh - bh + 1)), bw, bh))
    return out


def _roi_of(boxes):
    x0, y0 = min(b[0] for b in boxes), min(b[1] for b in boxes)
    return (x0, y0, max(b[0] + b[2] for b in boxes) - x0, max(b[1] + b[3] for b in boxes) - y0)


def _source_rects(case):
    """[(boxes, roi, pvp)] of a sort-last case; a cropped source stores the
    ``align``-pixel aligned columns around its region of interest."""
    out = []
    for i in range(case["n"]):
        boxes = _boxes(case, i)
        roi = _roi_of(boxes)
        if case.get("cropped", True):
            a = case.get("align", 4)
            x0 = roi[0] // a * a
            x1 = -(-(roi[0] + roi[2]) // a) * a
            pvp = (x0, roi[1], x1 - x0, roi[3])
        else:
            pvp = (0, 0, case["w"], case["h"])
        out.append((boxes, roi, pvp))
    return out


def _layer_rects(case):
    """[(pvp, roi)] of the blended layers: whole frames, or crops of which a
    border is not of interest."""
    W, H = case["w"], case["h"]
    if not case["cropped"]:
        return [((0, 0, W, H), (0, 0, W, H))] * case["n"]
    out = []
    for i in range(case["n"]):
        r = _layout(case, i)
        w, h = int(r.integers(W // 2, W + 1)), int(r.integers(H // 2, H + 1))
        x, y = int(r.integers(0, W - w + 1)), int(r.integers(0, H - h + 1))
        l, t, b = (int(v) for v in r.integers(0, 9, size=3))
        out.append(((x, y, w, h), (x + l, y + t, w - l, h - t - b)))
    return out


def _uneven(case):
    """[(mode, w, h, layers)] of a batch."""
    r = _layout(case, 0)
    out = []
    for k in range(case["n"]):
        w, h = (int(round(math.exp(r.uniform(math.log(16), math.log(case["side"]))))) for _ in range(2))
        out.append(("alpha" if k % 2 else "depth", w, h, int(r.integers(2, case["layers"] + 1))))
    return out


def _tile_rects(case):
    """The tiles of a sort-first frame: a grid whose borders the load moved."""
    r = _layout(case, 0)

    def cuts(size, n):
        step = size / n
        return [0] + [int(round((k + r.uniform(-0.3, 0.3)) * step)) for k in range(1, n)] + [size]
    xs, ys = cuts(case["w"], case["nx"]), cuts(case["h"], case["ny"])
    return [(xs[i], ys[j], xs[i + 1] - xs[i], ys[j + 1] - ys[j])
            for j in range(case["ny"]) for i in range(case["nx"])]


# ------------------------------------------------------------------ values


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _arena(shapes, dtype, align=64):
    """One zeroed buffer and views of it, each starting at a multiple of
    ``align`` elements."""
    at, offs = 0, []
    for s in shapes:
        offs.append(at)
        at += -(-max(1, math.prod(s)) // align) * align
    buf = torch.zeros(at, dtype=dtype, device="cuda")
    return buf, [buf[o:o + math.prod(s)].view(s) for o, s in zip(offs, shapes)]


def _paint_flat(rects, seed):
    """Flat polygons: one colour and one depth per part, later parts on top."""
    r = np.random.Generator(np.random.PCG64(seed))
    out = []
    for boxes, roi, pvp in rects:
        color = torch.zeros((pvp[3], pvp[2]), dtype=torch.int32, device="cuda")
        depth = torch.ones((pvp[3], pvp[2]), dtype=torch.float32, device="cuda")
        rgb = (r.integers(0, 1 << 24, size=len(boxes)) | (255 << 24)).astype(np.uint32).view(np.int32)
        z = r.random(len(boxes), dtype=np.float32)
        for (x, y, w, h), c, d in zip(boxes, rgb, z):
            sl = (slice(y - pvp[1], y - pvp[1] + h), slice(x - pvp[0], x - pvp[0] + w))
            color[sl] = int(c)
            depth[sl] = float(d)
        out.append((color, depth))
    return out


def _paint_shaded(rects, seed):
    """Ellipsoids with diffuse shading and their own depth, nearer ones in front."""
    r = np.random.Generator(np.random.PCG64(seed))
    out = []
    for boxes, roi, pvp in rects:
        color = torch.zeros((pvp[3], pvp[2]), dtype=torch.int32, device="cuda")
        depth = torch.ones((pvp[3], pvp[2]), dtype=torch.float32, device="cuda")
        for (x, y, w, h) in boxes:
            rgb, z0 = r.integers(64, 256, size=3), float(r.uniform(0.2, 0.9))
            u = (torch.arange(w, device="cuda", dtype=torch.float32) + 0.5) * (2.0 / w) - 1.0
            v = (torch.arange(h, device="cuda", dtype=torch.float32) + 0.5) * (2.0 / h) - 1.0
            z2 = 1.0 - u[None, :].square() - v[:, None].square()
            n = z2.clamp(min=0).sqrt()
            d = z0 - 0.1 * n
            light = (0.25 + 0.75 * (0.4 * u[None, :] - 0.3 * v[:, None] + 0.86 * n).clamp(0, 1))
            px = torch.full((h, w), -(1 << 24), dtype=torch.int32, device="cuda")      # alpha 255
            for k in range(3):
                px |= (light * float(rgb[k])).to(torch.int32) << (8 * k)
            sl = (slice(y - pvp[1], y - pvp[1] + h), slice(x - pvp[0], x - pvp[0] + w))
            hit = (z2 > 0) & (d < depth[sl])
            depth[sl] = torch.where(hit, d, depth[sl])
            color[sl] = torch.where(hit, px, color[sl])
        out.append((color, depth))
    return out


def _fill_layer(t, g, amax):
    """Premultiplied RGBA: alpha ~ U[0, amax], colour = alpha * U[0, 1)."""
    a = torch.rand(t.shape[:-1], generator=g, device="cuda") * amax
    t[..., :3] = torch.rand((*t.shape[:-1], 3), generator=g, device="cuda") * a[..., None]
    t[..., 3] = a


def _u32(t):
    return t.view(torch.uint32)


# ----------------------------------------------------------------- prepare


class _Codec:
    """Compress and decompress calls over planes [(int32 [h][w], mode)], planned once."""

    def __init__(self, planes):
        caps = [(ec.rle_max_size(t.shape[1], t.shape[0]),) for t, _ in planes]
        self.streams, bufs = _arena(caps, torch.uint8, 256)
        self.sizes = torch.zeros(len(planes), dtype=torch.int64, device="cuda")
        sizes = [s.view(torch.uint64) for s in self.sizes.split(1)]
        self.back, self.dec = _arena([t.shape for t, _ in planes], torch.int32)
        self.comp, _ = ec.prepare_rle_compress_batch([(_u32(t), m, None, b, s)
                                                      for (t, m), b, s in zip(planes, bufs, sizes)])
        self.decomp, _ = ec.prepare_rle_decompress_batch([(b, t.shape[1], t.shape[0], _u32(d), None)
                                                          for (t, _), b, d in zip(planes, bufs, self.dec)])


def _frame_out(case):
    return (torch.zeros((case["h"], case["w"]), dtype=torch.int32, device="cuda"),
            torch.zeros((case["h"], case["w"]), dtype=torch.float32, device="cuda"))


def prepare(case, seed):
    k = case["kind"]
    S = {"kind": k}
    if k in ("merge", "frame", "swap", "roi", "shaded", "yuv"):
        if k in ("swap", "roi"):
            case = dict(case, align=4, cropped=k == "swap")
        # (whole frames are searched, so where their geometry lies is free to follow the seed)
        rects = _source_rects(dict(case, layout=seed) if k == "roi" else case)
        src = (_paint_shaded if k in ("shaded", "yuv") else _paint_flat)(rects, seed)
    if k in ("merge", "swap", "roi"):
        S["images"] = [ec.Image(color=_u32(c), depth=d, pvp=pvp, roi=pvp if k == "roi" else roi)
                       for (c, d), (_, roi, pvp) in zip(src, rects)]
    if k in ("merge", "frame", "swap"):
        S["color"], S["depth"] = _frame_out(case)
    if k == "merge":
        S["winner"] = torch.zeros((case["h"], case["w"]), dtype=torch.int16, device="cuda") if case["winner"] else None
    elif k in ("frame", "shaded"):
        planes = [p for c, d in src for p in ((c, 2), (d.view(torch.int32), 1))]
        S["codec"], S["keep"] = _Codec(planes), planes
        if k == "frame":
            dec = S["codec"].dec
            S["images"] = [ec.Image(color=_u32(dec[2 * i]), depth=dec[2 * i + 1].view(torch.float32), pvp=pvp, roi=roi)
                           for i, (_, roi, pvp) in enumerate(rects)]
    elif k == "yuv":
        color = [c for c, _ in src]
        _, packed = _arena([ec.yuv_packed_shape(c.shape[1], c.shape[0]) for c in color], torch.int32)
        S["codec"] = _Codec([(p, 1) for p in packed])
        S["out"], views = _arena([c.shape for c in color], torch.int32)
        S["encode"] = ec.prepare_yuv_batch([(_u32(c), _u32(p), c.shape[1], c.shape[0])
                                            for c, p in zip(color, packed)], True)
        S["decode"] = ec.prepare_yuv_batch([(_u32(p), _u32(v), v.shape[1], v.shape[0])
                                            for p, v in zip(S["codec"].dec, views)], False)
        S["keep"] = [color, packed, views]
    elif k == "swap":
        S["plan"] = ec.Schedule("depth", case["algorithm"], S["images"], _u32(S["color"]), S["depth"])
    elif k == "roi":
        S["tile"] = case["tile"]
    elif k in ("over", "train"):
        dtype = torch.float16 if case["half"] else torch.float32
        g, rects = _generator(seed), _layer_rects(case)
        _, layers = _arena([(p[3], p[2], 4) for p, _ in rects], dtype)
        for t in layers:
            _fill_layer(t, g, case["amax"])
        S["images"] = [ec.Image(color=t, pvp=p, roi=r) for t, (p, r) in zip(layers, rects)]
        S["order"] = list(range(case["n"]))[::-1] if case["back"] else None
        S["out"] = torch.zeros((case["h"], case["w"], 4), dtype=dtype, device="cuda")
        S["left"] = torch.zeros((case["h"], case["w"]), dtype=torch.float32, device="cuda")
        if k == "train":
            S["w"] = torch.rand((case["h"], case["w"], 4), generator=g, device="cuda") * 2 - 1
            S["grad"], S["grads"] = _arena([t.shape for t in layers], dtype)
    elif k == "batch":
        g = _generator(seed)
        tiles = _uneven(case)
        D = [t for t in tiles if t[0] == "depth"]
        A = [t for t in tiles if t[0] == "alpha"]
        S["color"], oc = _arena([(h, w) for _, w, h, _ in D], torch.int32)
        S["depth"], od = _arena([(h, w) for _, w, h, _ in D], torch.float32)
        S["alpha"], oa = _arena([(h, w, 4) for _, w, h, _ in A], torch.float32)
        jobs, S["layers"] = [], []
        for k2, (mode, w, h, L) in enumerate(tiles):
            if mode == "depth":
                c, d = _flat_stack(L, w, h, g)
                imgs = [ec.Image(color=_u32(c[i]), depth=d[i]) for i in range(L)]
                jobs.append(ec.Job("depth", imgs, _u32(oc[k2 // 2]), od[k2 // 2]))
            else:
                t = torch.empty((L, h, w, 4), device="cuda")
                _fill_layer(t, g, 0.3)
                jobs.append(ec.Job("alpha", [ec.Image(color=t[i]) for i in range(L)], oa[k2 // 2]))
                S["layers"].append(t)
        S["plan"] = ec.Batch(jobs, config={})     # the tile shapes are stated, so every plan is the same one
    elif k == "tiles":
        g = _generator(seed)
        S["images"] = []
        for r in _tile_rects(case):
            if case["half"]:
                t = torch.rand((r[3], r[2], 4), generator=g, device="cuda").to(torch.float16)
            else:
                t = _u32(torch.randint(-(1 << 31), 1 << 31, (r[3], r[2]), generator=g, device="cuda", dtype=torch.int64)
                         .to(torch.int32))
            S["images"].append(ec.Image(color=t, pvp=r, roi=r))
        shape = (case["h"], case["w"], 4) if case["half"] else (case["h"], case["w"])
        S["out"] = torch.zeros(shape, dtype=torch.float16 if case["half"] else torch.int32, device="cuda")
    return S


def _flat_stack(L, w, h, g):
    """L layers of 12 flat rectangles over the background."""
    n = 12
    u = torch.rand((4, n, L, 1, 1), generator=g, device="cuda")
    bw, bh = (w * (0.125 + 0.21 * u[0])).ceil(), (h * (0.125 + 0.21 * u[1])).ceil()
    x0, y0 = (u[2] * (w - bw)).floor(), (u[3] * (h - bh)).floor()
    rgb = torch.randint(0, 1 << 24, (n, L, 1, 1), generator=g, device="cuda", dtype=torch.int32) | -(1 << 24)
    z = torch.rand((n, L, 1, 1), generator=g, device="cuda")
    xs, ys = torch.arange(w, device="cuda").float(), torch.arange(h, device="cuda").float()[:, None]
    c = torch.zeros((L, h, w), dtype=torch.int32, device="cuda")
    d = torch.ones((L, h, w), device="cuda")
    for k in range(n):
        m = ((xs >= x0[k]) & (xs < x0[k] + bw[k])) & ((ys >= y0[k]) & (ys < y0[k] + bh[k]))
        c = torch.where(m, rgb[k], c)
        d = torch.where(m, z[k], d)
    return c, d


# --------------------------------------------------------------------- run


def run(S):
    k = S["kind"]
    if k == "merge":
        roi = ec.composite_depth(S["images"], _u32(S["color"]), S["depth"], winner=S["winner"])
        return [S["color"], S["depth"].view(torch.int32), S["winner"], list(roi)]
    if k in ("frame", "shaded"):
        c = S["codec"]
        c.comp.run()
        c.decomp.run()
        out = [c.streams, c.sizes, c.back]
        if k == "frame":
            ec.composite_depth(S["images"], _u32(S["color"]), S["depth"])
            out += [S["color"], S["depth"].view(torch.int32)]
        return out
    if k == "yuv":
        c = S["codec"]
        S["encode"].run()
        c.comp.run()
        c.decomp.run()
        S["decode"].run()
        return [c.streams, c.sizes, c.back, S["out"]]
    if k == "over":
        ec.composite_alpha(S["images"], S["out"], order=S["order"], t_final=S["left"])
        return [S["out"], S["left"]]
    if k == "train":
        ec.composite_alpha_fwd_bwd(S["images"], S["out"], S["w"], S["grads"], order=S["order"], t_final=S["left"])
        return [S["out"], S["left"], S["grad"]]
    if k == "swap":
        S["plan"].run()
        return [S["color"], S["depth"].view(torch.int32)]
    if k == "batch":
        S["plan"].run()
        return [S["color"], S["depth"].view(torch.int32), S["alpha"]]
    if k == "tiles":
        out = S["out"]
        ec.assemble_tiles(S["images"], out if out.dim() == 3 else _u32(out))
        return out.view(torch.int16) if out.dim() == 3 else out
    rois, grids = ec.detect_roi(S["images"], S["tile"])
    return [rois, *grids[:60]]


# -------------------------------------------------------------------- work

# Bytes of a coded stream per byte of its pixels, as measured: flat polygons,
# shaded ones (a good part of a crop is background), and the latter's packed YUV.
_FLAT, _SHADED, _PACKED = 0.02, 0.27, 0.27


def work(case):
    k = case["kind"]
    if k in ("merge", "frame", "swap", "roi", "shaded", "yuv"):
        if k in ("swap", "roi"):
            case = dict(case, align=4, cropped=k == "swap")
        rects = _source_rects(case)
        stored = sum(p[2] * p[3] for _, _, p in rects)
        wanted = sum(max(0, r[2]) * max(0, r[3]) for _, r, _ in rects)
        frame = case["w"] * case["h"]
        if k == "merge":
            return {"bytes": 8 * wanted + (10 if case["winner"] else 8) * frame, "flops": 0}
        if k == "frame":
            return {"bytes": int(16 * stored * (1 + _FLAT)) + 8 * wanted + 8 * frame, "flops": 0}
        if k == "shaded":
            return {"bytes": int(16 * stored * (1 + _SHADED)), "flops": 0}
        if k == "yuv":                            # RGBA8 to 2 bytes a pixel, coded, and back
            return {"bytes": int(stored * 2 * (4 + 2 + 2 + 2 * _PACKED)), "flops": 0}
        if k == "swap":                           # each source read once, the frame written once
            return {"bytes": 8 * wanted + 8 * frame, "flops": 0}
        return {"bytes": 4 * case["n"] * frame, "flops": 0}
    if k in ("over", "train"):
        px = 8 if case["half"] else 16
        rects = _layer_rects(case)
        read = sum(r[2] * r[3] for _, r in rects)
        frame = case["w"] * case["h"]
        if k == "over":
            return {"bytes": px * read + (px + 4) * frame, "flops": 10 * read}
        grad = sum(p[2] * p[3] for p, _ in rects)
        return {"bytes": px * (read + grad) + (px + 4 + 16) * frame, "flops": 30 * read}
    if k == "batch":
        total = 0
        for mode, w, h, L in _uneven(case):
            total += (L + 1) * w * h * (8 if mode == "depth" else 16)
        return {"bytes": total, "flops": 0}
    return {"bytes": 2 * (8 if case["half"] else 4) * case["w"] * case["h"], "flops": 0}


# ------------------------------------------------------------------- exact


def _over64(S, layers, frame):
    """(out, transmittance, per-layer T) in 64 bits, front to back."""
    h, w = frame
    out = torch.zeros((h, w, 4), dtype=torch.float64, device="cuda")
    T = torch.ones((h, w, 1), dtype=torch.float64, device="cuda")
    for sl, c in layers:
        c = c.double()
        out[sl] += T[sl] * c
        T[sl] *= 1.0 - c[..., 3:]
    return out, T


def exact(case, seed):
    """Blended colours, transmittance and gradients in 64 bits.  The other
    outputs are whole numbers or copies of input words."""
    k = case["kind"]
    if k not in ("over", "train", "batch"):
        return None
    S = prepare(case, seed)
    if k == "batch":
        tiles = [t for t in _uneven(case) if t[0] == "alpha"]
        buf, outs = _arena([(h, w, 4) for _, w, h, _ in tiles], torch.float64)
        for o, t in zip(outs, S["layers"]):
            o.copy_(_over64(S, [((slice(None), slice(None)), c) for c in t], o.shape[:2])[0])
        return [None, None, buf]
    order = S["order"] or list(range(case["n"]))
    layers = []
    for i in order:
        im = S["images"][i]
        (px, py, _, _), (x, y, w, h) = im.pvp, im.roi
        layers.append(((slice(y, y + h), slice(x, x + w)), im.color[y - py:y - py + h, x - px:x - px + w]))
    out, T = _over64(S, layers, (case["h"], case["w"]))
    left = T[..., 0].clone()
    if k == "over":
        return [out, left]
    # back to front: T before each layer, and A = sum over the layers behind of
    # w . c times the transmittance between
    w64 = S["w"].double()
    grad, grads = _arena([t.shape for t in S["grads"]], torch.float64)
    A = torch.zeros_like(T)
    for i, (sl, c) in zip(order[::-1], layers[::-1]):
        c = c.double()
        through = 1.0 - c[..., 3:]
        T[sl] /= through                          # alpha <= 0.3: no cancellation
        im = S["images"][i]
        (px, py, _, _), (x, y, w, h) = im.pvp, im.roi
        v = grads[i][y - py:y - py + h, x - px:x - px + w]
        v.copy_(T[sl] * w64[sl])
        v[..., 3:] -= T[sl] * A[sl]
        A[sl] = (w64[sl] * c).sum(-1, keepdim=True) + through * A[sl]
    return [out, left, grad]
