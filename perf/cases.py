"""Performance cases of the variable-rate (JPEG) texture path.

Each case is one pass that a renderer (or a trainer, for the float chain) makes through the
package's public calls, on seeded inputs made here with torch: value-noise textures, encoded
as baseline JPEG with mip chains, and deferred G-buffers of a ground plane of textured cells
under screen-space quads (the benchmark's scene, with sizes from the benchmark and the tests).

    listed()              the named cases
    draw(rng)             one more case of the same ranges
    prepare(case, seed)   what a program holds before the pass: a context with its textures
                          uploaded, G-buffers, output buffers, captured graphs
    run(state)            one pass
    work(case)            the bytes and operations a pass cannot do without
    exact(case, seed)     the float chain's outputs in 64 bits
"""

from __future__ import annotations

import functools
import math
import random
from types import SimpleNamespace

import numpy as np
import torch
import torch.nn.functional as F

import paper_2510_08166_gb300 as jt

DEVICE = "cuda:0"
FILTERS = {"nearest": jt.FILTER_NEAREST, "bilinear": jt.FILTER_BILINEAR, "clamped": jt.FILTER_BILINEAR_CLAMP}

# A frame case: `textures` textures with sides drawn from lo, 2 lo, .. hi (plus `odd` texels, so
# that sides stop being powers of two), qualities 50..95, full mip chains; `views` views of
# width x height. mode: "calls" (mark, decode, colorize), "frame" (one batched call) or "graph"
# (a captured frame, replayed). form: how the textures are stored and indexed.
FRAME = {"kind": "frame", "textures": 24, "lo": 512, "hi": 2048, "odd": 0, "sampling": "420", "form": "standard",
         "huffman": "standard", "views": 1, "filter": "bilinear", "mode": "frame", "tuned": False}


def listed():
    return [
        # the smallest call: a texture preview or a unit of a tool, three calls on a 256 x 256
        # view of one 512^2 texture; latency and launches
        {**FRAME, "name": "preview_256_calls", "textures": 1, "lo": 512, "hi": 512, "width": 256, "height": 256,
         "filter": "nearest", "mode": "calls"},
        # the ordinary frame of a game or viewer: 1080p, mips, eager batched call
        {**FRAME, "name": "frame_1080p", "width": 1920, "height": 1080},
        # the headline: 4K, 64 textures of 1024..4096, a captured frame with the launch shape
        # that the autotuner picks for it
        {**FRAME, "name": "frame_4k_graph", "textures": 64, "lo": 1024, "hi": 4096, "width": 3840, "height": 2160,
         "mode": "graph", "tuned": True},
        # textures in the paper's compact random-access form, its clamped filter, 1440p
        {**FRAME, "name": "frame_1440p_compact", "form": "compact", "width": 2560, "height": 1440,
         "filter": "clamped"},
        # data-unit starts stored beside the index, 1080p graph
        {**FRAME, "name": "frame_1080p_units", "form": "units", "width": 1920, "height": 1080, "mode": "graph"},
        # lower levels by reduced decode instead of stored mips (the mip alternative), 1440p
        {**FRAME, "name": "frame_1440p_reduced", "form": "reduced", "textures": 16, "width": 2560, "height": 1440},
        # odd sizes throughout: 4:4:4 and 4:2:0 textures whose sides are no powers of two, each
        # with Huffman tables of its own (as an optimising encoder writes them), odd view
        {**FRAME, "name": "frame_odd_own_tables", "odd": 37, "sampling": "mixed", "huffman": "own", "textures": 12,
         "width": 1367, "height": 769, "mode": "calls"},
        # a head-mounted display: both eyes in one captured frame, clamped filter
        {**FRAME, "name": "vr_pair_graph", "views": 2, "width": 2064, "height": 2208, "filter": "clamped",
         "mode": "graph"},
        # a turning camera with the cross-frame block cache: six directions 6 degrees apart,
        # one captured frame each (the first one returns from the last, so it misses most)
        {**FRAME, "name": "motion_1080p_cache", "kind": "motion", "directions": 6, "width": 1920, "height": 1080,
         "mode": "graph"},
        # whole textures to pixels (export, baking, a full decode): one pixel per texel of eight
        # 4096^2 textures at quality 90, half of them 4:4:4; every MCU needed
        {"kind": "bake", "name": "bake_8x4096", "textures": 8, "size": 4096, "quality": 90, "sampling": "mixed"},
        # differentiable colourise, forward and backward: sixteen 2048^2 coefficient textures,
        # a 1080p ground plane without mips
        {"kind": "float", "name": "float_1080p_train", "textures": 16, "size": 2048, "width": 1920, "height": 1080},
        # the scene rasterised on the GPU at 4K: 64 textures, 200 quads
        {"kind": "raster", "name": "raster_4k", "textures": 64, "quads": 200, "width": 3840, "height": 2160,
         "mips": True},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _screen(rng, lo, hi):
    """Width and height of a view with sides of lo..hi pixels, odd ones among them."""
    w = _log(rng, lo, hi)
    h = max(lo * 9 // 16, int(w * rng.choice([9 / 16, 10 / 16, 3 / 4, 1.0])))
    return w, min(h, 2208)


def draw(rng):
    kind = rng.choice(["frame"] * 6 + ["motion", "bake", "float", "raster"])
    if kind in ("frame", "motion"):
        w, h = _screen(rng, 200, 3840 if kind == "frame" else 2200)
        lo = rng.choice([256, 512, 1024])
        c = {**FRAME, "kind": kind, "textures": _log(rng, 1, 32), "lo": lo, "hi": lo * rng.choice([1, 2, 4]),
             "odd": rng.choice([0, 0, rng.randrange(1, 99)]), "sampling": rng.choice(["420", "420", "444", "mixed"]),
             "form": rng.choice(["standard", "standard", "compact", "units", "reduced"]),
             "huffman": rng.choice(["standard", "standard", "own"]), "width": w, "height": h,
             "filter": rng.choice(["nearest", "bilinear", "bilinear", "clamped"])}
        if kind == "motion":
            return {**c, "directions": rng.randrange(3, 7), "mode": "graph"}
        mode = rng.choice(["calls", "frame", "graph"])
        return {**c, "mode": mode, "views": 1 if mode == "calls" else rng.choice([1, 1, 2, 3]),
                "tuned": rng.choice([False, False, True])}
    if kind == "bake":
        return {"kind": "bake", "textures": rng.randrange(1, 9), "size": _log(rng, 250, 4096),
                "quality": rng.randrange(50, 96), "sampling": rng.choice(["420", "444", "mixed"])}
    if kind == "float":
        w, h = _screen(rng, 128, 1920)
        return {"kind": "float", "textures": rng.randrange(1, 17), "size": 16 * _log(rng, 8, 128), "width": w,
                "height": h}
    w, h = _screen(rng, 200, 3840)
    return {"kind": "raster", "textures": _log(rng, 1, 128), "quads": rng.choice([0, _log(rng, 4, 1000)]), "width": w,
            "height": h, "mips": rng.random() < 0.8}


def work(case):
    px = case.get("width", 0) * case.get("height", 0)
    kind = case["kind"]
    if kind in ("frame", "motion"):
        # G-buffer read once (11 B a pixel), RGBA8 written once; the needed MCUs' streams and
        # index entries: on these mipmapped scenes about one MCU per 300 pixels, 42 B each
        n = px * case["views"] * case.get("directions", 1)
        return {"bytes": 15.0 * n + 42.0 * (n / 300 + 64), "flops": 0.0}
    if kind == "bake":
        n = case["textures"] * case["size"] ** 2
        return {"bytes": 15.0 * n + 0.25 * n, "flops": 0.0}
    if kind == "float":
        # forward: G-buffer, the coefficients of the MCUs the pixels touch (at most all, at
        # most about one per nine pixels), the frame written; backward: G-buffer and frame
        # gradient read, the dense gradient written
        mcus = case["textures"] * (case["size"] // 16) ** 2
        need = min(mcus, px / 9 + 64)
        return {"bytes": 2 * 11.0 * px + 24.0 * px + 1536.0 * need + 1536.0 * mcus,
                "flops": need * 2 * 6 * 2 * 8 * 64.0 + 2 * 24.0 * px}
    return {"bytes": 11.0 * px, "flops": 60.0 * px}


# ---------------------------------------------------------------------------------------
# Textures
# ---------------------------------------------------------------------------------------

def _noise_image(gen, h, w):
    """RGB float [h, w, 3] in 0..255: value noise of many octaves mixed by a random matrix, with
    two dozen solid rectangles over it."""
    acc = torch.zeros((1, 3, h, w), device=DEVICE)
    spacing = float(max(h, w))
    while spacing >= 2:
        lat = torch.rand((1, 3, max(2, round(h / spacing) + 1), max(2, round(w / spacing) + 1)), device=DEVICE,
                         generator=gen) - 0.5
        acc += min(1.0, math.sqrt(spacing / 256)) * F.interpolate(lat, size=(h, w), mode="bilinear",
                                                                  align_corners=False)
        spacing /= 2
    mix = torch.rand((3, 3), device=DEVICE, generator=gen) + 0.3 * torch.eye(3, device=DEVICE)
    img = (acc[0].permute(1, 2, 0).reshape(-1, 3) @ mix).reshape(h, w, 3) * 60 + 128
    r = random.Random(int(torch.randint(1 << 30, (1,), device=DEVICE, generator=gen)))
    for _ in range(24):
        y, x = r.randrange(h), r.randrange(w)
        dy, dx = 1 + r.randrange(max(1, h // 8)), 1 + r.randrange(max(1, w // 8))
        img[y:y + dy, x:x + dx] = torch.tensor([r.randrange(256) for _ in range(3)], device=DEVICE, dtype=img.dtype)
    return img.clamp(0, 255)


def _half(img):
    """Next mip level: 2x2 box filter, sides at least 1."""
    h, w = max(1, img.shape[0] // 2), max(1, img.shape[1] // 2)
    y = torch.arange(h, device=DEVICE) * (2 if img.shape[0] > 1 else 1)
    x = torch.arange(w, device=DEVICE) * (2 if img.shape[1] > 1 else 1)
    y1, x1 = (y + 1).clamp(max=img.shape[0] - 1), (x + 1).clamp(max=img.shape[1] - 1)
    a, b = img[y], img[y1]
    return (a[:, x] + a[:, x1] + b[:, x] + b[:, x1]) * 0.25


@functools.lru_cache(maxsize=None)
def _zigzag():
    """Natural index of each zig-zag position."""
    order = sorted(((r, c) for r in range(8) for c in range(8)),
                   key=lambda p: (p[0] + p[1], p[0] if (p[0] + p[1]) & 1 else p[1]))
    return [r * 8 + c for r, c in order]


def _dct_matrix(dtype):
    k, n = torch.meshgrid(torch.arange(8, dtype=torch.float64), torch.arange(8, dtype=torch.float64), indexing="ij")
    d = 0.5 * torch.cos((2 * n + 1) * k * math.pi / 16)
    d[0] *= math.sqrt(0.5)
    return d.to(DEVICE, dtype)


# The example quantisation tables of the JPEG standard (luma, chroma), natural order.
_QT = ([16, 11, 10, 16, 24, 40, 51, 61, 12, 12, 14, 19, 26, 58, 60, 55, 14, 13, 16, 24, 40, 57, 69, 56, 14, 17, 22, 29,
        51, 87, 80, 62, 18, 22, 37, 56, 68, 109, 103, 77, 24, 35, 55, 64, 81, 104, 113, 92, 49, 64, 78, 87, 103, 121,
        120, 101, 72, 92, 95, 98, 112, 100, 103, 99],
       [17, 18, 24, 47, 99, 99, 99, 99, 18, 21, 26, 66, 99, 99, 99, 99, 24, 26, 56, 99, 99, 99, 99, 99, 47, 66, 99, 99,
        99, 99, 99, 99] + [99] * 32)


def _quant_tables(quality):
    s = 5000 // quality if quality < 50 else 200 - 2 * quality
    return np.clip((np.array(_QT) * s + 50) // 100, 1, 255).astype(np.uint16)


def _all_ac():
    return [(r << 4) | s for r in range(16) for s in range(1, 11)] + [0x00, 0xF0]


@functools.lru_cache(maxsize=None)
def _standard_huffman():
    """The typical tables of the JPEG standard: (bits, symbols) of DC luma, AC luma, DC chroma,
    AC chroma. The longest codes of an AC table are its remaining symbols in order."""
    dc = list(range(12))
    luma = bytes.fromhex("0102030004110512213141061351610722711432"
                         "8191a1082342b1c11552d1f02433627282")
    chroma = bytes.fromhex("0001020311040521310612415107617113223281081442"
                           "91a1b1c109233352f0156272d10a162434e125f1")

    def rest(head):
        return list(head) + sorted(set(_all_ac()) - set(head))

    return (([0, 1, 5, 1, 1, 1, 1, 1, 1, 0, 0, 0, 0, 0, 0, 0], dc),
            ([0, 2, 1, 3, 3, 2, 4, 3, 5, 5, 4, 4, 0, 0, 1, 0x7D], rest(luma)),
            ([0, 3, 1, 1, 1, 1, 1, 1, 1, 1, 1, 0, 0, 0, 0, 0], dc),
            ([0, 2, 1, 2, 4, 4, 3, 4, 7, 5, 4, 4, 0, 1, 2, 0x77], rest(chroma)))


def _own_huffman(counts):
    """Tables fitted to symbol counts [4][256]: each symbol's code takes ceil(-log2 p) bits, with
    every symbol of the class kept codable within 14 bits."""
    specs = []
    for t in range(4):
        syms = list(range(12)) if t % 2 == 0 else _all_ac()
        total, eps = max(1, int(counts[t].sum())), 2.0 ** -13
        p = {s: (counts[t][s] / total + eps) / (1 + (len(syms) + 1) * eps) for s in syms}
        length = {s: max(1, math.ceil(-math.log2(p[s]))) for s in syms}
        order = sorted(syms, key=lambda s: (length[s], s))
        specs.append(([sum(length[s] == i for s in syms) for i in range(1, 17)], order))
    return tuple(specs)


def _codes(spec):
    """(code [256], length [256]) of one table's canonical code."""
    code, length, c, k = np.zeros(256, np.int64), np.zeros(256, np.int64), 0, 0
    for n, count in enumerate(spec[0], 1):
        for _ in range(count):
            code[spec[1][k]], length[spec[1][k]] = c, n
            c, k = c + 1, k + 1
        c <<= 1
    return code, length


def _blocks(img, sampling):
    """Data units [nmcu, ndu, 8, 8] of an RGB image (level-shifted YCbCr, edges replicated, in
    MCU order) and the MCU grid."""
    mw = 16 if sampling == 420 else 8
    my, mx = -(-img.shape[0] // mw), -(-img.shape[1] // mw)
    m = torch.tensor([[0.299, -0.168736, 0.5], [0.587, -0.331264, -0.418688], [0.114, 0.5, -0.081312]], device=DEVICE,
                     dtype=img.dtype)
    ycc = (img.reshape(-1, 3) @ m).reshape(img.shape)
    y = torch.arange(my * mw, device=DEVICE).clamp(max=img.shape[0] - 1)
    x = torch.arange(mx * mw, device=DEVICE).clamp(max=img.shape[1] - 1)
    ycc = ycc[y][:, x] - torch.tensor([128.0, 0, 0], device=DEVICE, dtype=img.dtype)
    if sampling == 444:
        return ycc.reshape(my, 8, mx, 8, 3).permute(0, 2, 4, 1, 3).reshape(my * mx, 3, 8, 8), mx, my
    luma = ycc[..., 0].reshape(my, 2, 8, mx, 2, 8).permute(0, 3, 1, 4, 2, 5).reshape(my * mx, 4, 8, 8)
    ch = ycc[..., 1:].reshape(my * 8, 2, mx * 8, 2, 2).mean(dim=(1, 3))
    ch = ch.reshape(my, 8, mx, 8, 2).permute(0, 2, 4, 1, 3).reshape(my * mx, 2, 8, 8)
    return torch.cat([luma, ch], 1), mx, my


def _quantised(img, sampling, qt):
    """Quantised coefficients [nmcu, ndu, 64] int64 (natural order) and the MCU grid."""
    blk, mx, my = _blocks(img, sampling)
    d = _dct_matrix(blk.dtype)
    c = (d @ blk @ d.T).reshape(blk.shape[0], blk.shape[1], 64)
    q = torch.tensor(qt.astype(np.float32), device=DEVICE)
    nl = blk.shape[1] - 2
    q = torch.cat([q[:1].expand(nl, 64), q[1:].expand(2, 64)])
    return torch.round(c / q).clamp(-1023, 1023).long(), mx, my


def _put(words, start, value, length):
    """Adds `length`-bit values at bit positions `start` (most significant first) of the 32-bit
    words; the values' bits do not overlap."""
    w, o = start >> 5, start & 31
    for j in range(3):
        sh = length - (32 * (j + 1) - o)
        part = torch.where(sh >= 0, value >> sh.clamp(min=0, max=62), value << (-sh).clamp(min=0, max=32)) & 0xFFFFFFFF
        words.scatter_add_(0, w + j, part)


def _encode(images, quality, sampling, form, huffman):
    """The levels of one texture, coded together (one stream each): what Context.upload,
    upload_compact and set_du_offsets take."""
    qt = _quant_tables(quality)
    parts = [_quantised(img, sampling, qt) for img in images]
    q = torch.cat([p[0] for p in parts])
    nmcu, ndu, _ = q.shape
    nl = ndu - 2
    first = np.cumsum([0] + [p[0].shape[0] for p in parts])  # first MCU of each level, and the end
    heads = torch.tensor(first[:-1], device=DEVICE)
    z = q[:, :, _zigzag()]
    compact = form == "compact"
    cat = torch.tensor([0] + [int(v).bit_length() for v in range(1, 4097)], device=DEVICE)

    # DC differences and each MCU's predictors (zero at the head of a level)
    dc = z[:, :, 0]
    prev = torch.zeros_like(dc)
    prev[1:, 0] = dc[:-1, nl - 1]
    prev[1:, nl:] = dc[:-1, nl:]
    prev[heads] = 0
    prev[:, 1:nl] = dc[:, :nl - 1]
    pred = prev[:, [0, nl, nl + 1]]
    diff = dc - prev
    dcs = cat[diff.abs()]
    cls = torch.zeros(ndu, dtype=torch.long, device=DEVICE)
    cls[nl:] = 1

    # AC symbols of the non-zero coefficients
    zf = z.reshape(nmcu * ndu, 64)
    nz = zf != 0
    nz[:, 0] = False
    pos = torch.arange(64, device=DEVICE)
    last = torch.where(nz, pos, 0).cummax(1).values
    u, k = nz.nonzero(as_tuple=True)
    run = k - last[u, k - 1] - 1
    v = zf[u, k]
    s = cat[v.abs()]
    ucls = cls[u % ndu]
    sym = ((run & 15) << 4) | s
    eob = last[:, 63] < 63

    tables = _standard_huffman()
    if huffman == "own":
        counts = np.zeros((4, 256), np.int64)
        for c in range(2):
            counts[2 * c] = torch.bincount(dcs[:, cls == c].flatten(), minlength=256).cpu().numpy()
            counts[2 * c + 1] = torch.bincount(sym[ucls == c], minlength=256).cpu().numpy()
            counts[2 * c + 1][0] += int(eob.reshape(nmcu, ndu)[:, cls == c].sum())
            counts[2 * c + 1][0xF0] += int((run >> 4)[ucls == c].sum())
        tables = _own_huffman(counts)
    codes = [_codes(t) for t in tables]
    code = torch.tensor(np.stack([c for c, _ in codes]), device=DEVICE)
    clen = torch.tensor(np.stack([n for _, n in codes]), device=DEVICE)
    tac = 2 * ucls + 1
    zcode, zlen = code[tac, 0xF0], clen[tac, 0xF0]
    nzrl = run >> 4

    # bit lengths per slot: DC, 63 AC positions (with the runs of 16 before them), end of block
    lens = torch.zeros((nmcu, ndu, 65), dtype=torch.long, device=DEVICE)
    has_dc = torch.ones(ndu, dtype=torch.bool, device=DEVICE)
    if compact:  # the first luma and the chroma DCs are stored apart
        has_dc[0] = has_dc[nl] = has_dc[nl + 1] = False
    dlen = clen[(2 * cls).expand(nmcu, ndu), dcs]
    lens[:, :, 0] = torch.where(has_dc, dlen + dcs, 0)
    lens.view(-1, 65)[u, k] = clen[tac, sym] + s + nzrl * zlen
    lens.view(-1, 65)[:, 64] = torch.where(eob, clen[2 * cls + 1, 0].repeat(nmcu), 0)
    flat = lens.view(nmcu, ndu * 65)
    inside = flat.cumsum(1) - flat
    bits = flat.sum(1)
    room = (bits + 7) // 8 * 8 if compact else bits
    # every level's stream starts on a word of its own
    ends = torch.cat([room.new_zeros(1), room.cumsum(0)])[torch.tensor(first, device=DEVICE)].tolist()
    total = [b - a for a, b in zip(ends, ends[1:])]
    origin = np.cumsum([0] + [(t + 31) // 32 * 32 for t in total])
    shift = torch.repeat_interleave(torch.tensor(origin[:-1] - np.array(ends[:-1]), device=DEVICE),
                                    torch.tensor(np.diff(first), device=DEVICE))
    base = room.cumsum(0) - room + shift
    start = (base[:, None] + inside).view(nmcu * ndu, 65)

    words = torch.zeros(int(origin[-1]) // 32 + 4, dtype=torch.long, device=DEVICE)
    mag = diff + torch.where(diff < 0, (1 << dcs) - 1, 0)
    dval = (code[(2 * cls).expand(nmcu, ndu), dcs] << dcs) | mag
    on = has_dc.expand(nmcu, ndu).reshape(-1)
    _put(words, start[on, 0], dval.reshape(-1)[on], lens.view(-1, 65)[on, 0])
    at = start[u, k]
    for i in range(3):
        m = nzrl > i
        _put(words, at[m] + i * zlen[m], zcode[m], zlen[m])
    _put(words, at + nzrl * zlen, (code[tac, sym] << s) | (v + torch.where(v < 0, (1 << s) - 1, 0)),
         clen[tac, sym] + s)
    e = eob.nonzero().flatten()
    ecls = 2 * cls[e % ndu] + 1
    _put(words, start[e, 64], code[ecls, 0], clen[ecls, 0])
    if compact:
        _put(words, base + bits, (1 << (room - bits)) - 1, room - bits)
    data = torch.stack([(words >> n) & 255 for n in (24, 16, 8, 0)], 1).to(torch.uint8).flatten().cpu().numpy()

    hb, hv = np.zeros((4, 16), np.uint8), np.zeros((4, 256), np.uint8)
    for t, (b, sy) in enumerate(tables):
        hb[t], hv[t, :len(sy)] = b, sy
    base, pred, dc3 = base.cpu().numpy(), pred.cpu().numpy(), dc[:, [0, nl, nl + 1]].cpu().numpy()
    units = inside.view(nmcu, ndu, 65)[:, 1:, 0].to(torch.int32).cpu().numpy().astype(np.uint16)
    levels = []
    for i, img in enumerate(images):
        m, o = slice(first[i], first[i + 1]), int(origin[i])
        scan = data[o // 8:o // 8 + (total[i] + 7) // 8]
        enc = SimpleNamespace(width=img.shape[1], height=img.shape[0], sampling=sampling, mcus_x=parts[i][1],
                              mcus_y=parts[i][2], scan=scan, scan_bits=total[i], qt=qt, huff_bits=hb, huff_vals=hv)
        if compact:
            enc.compact = _compact_tables(scan, (base[m] - o) // 8, dc3[m])
        else:
            enc.index = np.zeros(m.stop - m.start, np.dtype([("bit_offset", "<u4"), ("dc_pred", "<i2", (3,))]))
            enc.index["bit_offset"] = base[m] - o
            enc.index["dc_pred"] = pred[m]
            enc.du_offsets = units[m]
        levels.append(enc)
    return levels


def _compact_tables(scan, starts, dcs):
    """The compact form's side tables: two-level byte offsets and 36-bit DC records."""
    n = len(starts)
    ng = (n + 8) // 9
    rows = np.zeros((ng, 9), np.int64)
    rows.reshape(-1)[:n] = starts
    rel = np.maximum(rows[:, 1:] - rows[:, :1], 0).astype(np.uint16)
    d = (dcs & 0xFFF).astype(np.uint64)
    val = d[:, 0] | (d[:, 1] << np.uint64(12)) | (d[:, 2] << np.uint64(24))
    b = 36 * np.arange(n, dtype=np.uint64)
    o, w = b & np.uint64(31), (b >> np.uint64(5)).astype(np.int64)
    rec = np.zeros((36 * n + 31) // 32 + 1, np.uint64)
    np.add.at(rec, w, (val << o) & np.uint64(0xFFFFFFFF))
    np.add.at(rec, w + 1, val >> (np.uint64(32) - o))
    return SimpleNamespace(scan=scan, abs=rows[:, 0].astype(np.uint32), rel=rel.reshape(-1),
                           dc=rec[:(36 * n + 31) // 32].astype(np.uint32))


def _texture_draws(case, rng):
    """(side, quality, sampling) of each texture of a frame case."""
    steps = int(round(math.log2(case["hi"] / case["lo"]))) + 1
    out = []
    for t in range(case["textures"]):
        side = (case["lo"] << rng.randrange(steps)) + case["odd"]
        samp = {"420": 420, "444": 444, "mixed": 444 if t % 2 else 420}[case["sampling"]]
        out.append((side, side if not case["odd"] else side - case["odd"] // 2, 50 + rng.randrange(46), samp))
    return out


def _upload_textures(ctx, case, rng, gen):
    """Uploads the case's textures with their mip chains; returns sizes and level counts."""
    sizes, nlevels = [], []
    for t, (w, h, quality, sampling) in enumerate(_texture_draws(case, rng)):
        chain = [_noise_image(gen, h, w)]
        while max(chain[-1].shape[:2]) > 1:
            chain.append(_half(chain[-1]))
        # reduced form: every third level is stored, the two after it are decoded from its
        # lowest frequencies
        stored = [l for l in range(len(chain)) if case["form"] != "reduced" or l % 3 == 0]
        coded = _encode([chain[l] for l in stored], quality, sampling, case["form"], case["huffman"])
        for l in range(len(chain)):
            if l not in stored:
                ctx.add_reduced_level(t, l - l % 3, l % 3, l)
            elif case["form"] == "compact":
                ctx.upload_compact(t, l, coded[stored.index(l)])
            else:
                enc = coded[stored.index(l)]
                ctx.upload(t, l, enc)
                if case["form"] == "units":
                    ctx.set_du_offsets(t, l, enc.du_offsets)
        sizes.append((w, h))
        nlevels.append(len(chain))
    return sizes, nlevels


# ---------------------------------------------------------------------------------------
# G-buffers
# ---------------------------------------------------------------------------------------

def _pixels(width, height):
    y, x = torch.meshgrid(torch.arange(height, device=DEVICE, dtype=torch.float64) + 0.5,
                          torch.arange(width, device=DEVICE, dtype=torch.float64) + 0.5, indexing="ij")
    return x, y


def _rotation(yaw, pitch):
    cp, sp, cy, sy = (f(math.radians(a)) for a in (pitch, yaw) for f in (math.cos, math.sin))
    rx, ry = np.array([[1, 0, 0], [0, cp, -sp], [0, sp, cp]]), np.array([[cy, 0, sy], [0, 1, 0], [-sy, 0, cy]])
    return ry @ rx


def _ground_uv(px, py, width, height, cam, rot, vfov):
    """uv = world (x, z) / 2 of the ground point behind pixel coordinates, and where there is one."""
    th = math.tan(math.radians(vfov) / 2)
    sx, sy = (px * (2 / width) - 1) * th * width / height, (1 - py * (2 / height)) * th
    d = [rot[i][0] * sx + rot[i][1] * sy - rot[i][2] for i in range(3)]
    ok = d[1] < -1e-9
    t = -cam[1] / torch.where(ok, d[1], -1.0)
    return (cam[0] + t * d[0]) / 2, (cam[2] + t * d[2]) / 2, ok & (t <= 600)


def _mip(du, dv, tex, sizes, nlevels):
    tw, th = (torch.tensor([s[i] for s in sizes], device=DEVICE, dtype=torch.float64)[tex] for i in (0, 1))
    top = torch.tensor(nlevels, device=DEVICE)[tex] - 1
    rho = torch.stack([torch.hypot(a * tw, b * th) for a, b in zip(du, dv)]).amax(0)
    m = torch.floor(torch.log2(rho.clamp(min=1e-9, max=1e9)) + 0.5).long()
    return torch.minimum(m.clamp(min=0), top)


def _scene_gbuffer(width, height, sizes, nlevels, seed, cam=(0.0, 1.7, 0.0), yaw=20.0, pitch=-25.0, vfov=60.0,
                   quads=200, shift=0.0, mips=True):
    """Ground plane of 2 m cells, each with a texture and an offset of its own, under
    screen-space quads; mip level from the texel footprint of a pixel."""
    rot = _rotation(yaw, pitch)
    px, py = _pixels(width, height)
    u, v, ok = _ground_uv(px, py, width, height, cam, rot, vfov)
    cell = torch.floor(u).long() * 73856093 ^ torch.floor(v).long() * 19349663 ^ (seed * 2654435761 & 0xFFFFFFFF)
    cell = cell * 6364136223846793005 + 1442695040888963407
    cell = (cell >> 17) ^ cell
    tex = ((cell >> 40) & 0xFFFF) % len(sizes)
    lod = torch.zeros_like(tex)
    if mips:
        ends = [_ground_uv(px + dx, py + dy, width, height, cam, rot, vfov)
                for dx, dy in ((-0.5, 0), (0.5, 0), (0, -0.5), (0, 0.5))]
        lod = _mip([ends[1][0] - ends[0][0], ends[3][0] - ends[2][0]],
                   [ends[1][1] - ends[0][1], ends[3][1] - ends[2][1]], tex, sizes, nlevels)
        whole = ends[0][2] & ends[1][2] & ends[2][2] & ends[3][2]
        lod = torch.where(whole, lod, torch.tensor(nlevels, device=DEVICE)[tex] - 1)
    u, v = u + ((cell >> 8) & 0xFFFF) / 65536.0, v + ((cell >> 24) & 0xFFFF) / 65536.0
    zero = torch.zeros_like(u)
    u, v = torch.where(ok, u, zero), torch.where(ok, v, zero)
    tex, lod = torch.where(ok, tex, 0xFFFF), torch.where(ok, lod, 0)

    r = random.Random(seed ^ 0x51)
    for _ in range(quads):
        cx, cy = (r.random() + shift) * width, r.random() * height
        hw, hh, ang = (0.02 + 0.06 * r.random()) * height, (0.02 + 0.06 * r.random()) * height, r.uniform(0, math.pi)
        pers, rep, ou, ov, t = r.uniform(-0.3, 0.3), r.uniform(0.5, 2), r.random(), r.random(), r.randrange(len(sizes))
        rad = math.hypot(hw, hh)
        x0, x1 = max(0, int(cx - rad)), min(width, int(cx + rad) + 1)
        y0, y1 = max(0, int(cy - rad)), min(height, int(cy + rad) + 1)
        if x0 >= x1 or y0 >= y1:
            continue
        ca, sa = math.cos(ang), math.sin(ang)

        def local(x, y):
            a, b = x - cx, y - cy
            s, q = (a * ca + b * sa) / hw, (b * ca - a * sa) / hh
            w = 1 + pers * s
            return ou + rep * s / w, ov + rep * q / w, (s.abs() <= 1) & (q.abs() <= 1)

        x, y = px[y0:y1, x0:x1], py[y0:y1, x0:x1]
        qu, qv, inside = local(x, y)
        tq = torch.full_like(tex[y0:y1, x0:x1], t)
        lq = torch.zeros_like(tq)
        if mips:
            ends = [local(x + dx, y + dy) for dx, dy in ((-0.5, 0), (0.5, 0), (0, -0.5), (0, 0.5))]
            lq = _mip([ends[1][0] - ends[0][0], ends[3][0] - ends[2][0]],
                      [ends[1][1] - ends[0][1], ends[3][1] - ends[2][1]], tq, sizes, nlevels)
        for dst, src in ((u, qu), (v, qv), (tex, tq), (lod, lq)):
            dst[y0:y1, x0:x1] = torch.where(inside, src, dst[y0:y1, x0:x1])
    return _gbuffer(torch.stack([u, v], -1), tex, lod)


def _gbuffer(uv, tex, lod):
    tex = torch.where(tex > 32767, tex - 65536, tex).to(torch.int16)
    return uv.float().contiguous(), tex.contiguous(), lod.to(torch.uint8).contiguous()


def _affine_gbuffer(width, height, seed):
    """A texture turned and scaled over the view, level 0."""
    r = random.Random(seed)
    a, s = math.radians(r.uniform(5, 40)), r.uniform(1.1, 1.5)
    px, py = _pixels(width, height)
    x, y = px / width * s, py / height * s
    uv = torch.stack([x * math.cos(a) - y * math.sin(a), x * math.sin(a) + y * math.cos(a)], -1)
    zero = torch.zeros((height, width), dtype=torch.long, device=DEVICE)
    return _gbuffer(uv, zero, zero)


def _pose(case, seed, view):
    """Camera of a frame case's view: a pair of eyes 0.064 m apart when there are two or more."""
    r = random.Random(seed)
    cam, yaw, pitch = (r.uniform(-5, 5), 1.7, r.uniform(-5, 5)), r.uniform(0, 360), r.uniform(-35, -20)
    if case["views"] == 1:
        return {"cam": cam, "yaw": yaw, "pitch": pitch}
    side = 0.064 * (view - 0.5)
    right = (math.cos(math.radians(yaw)), 0.0, -math.sin(math.radians(yaw)))
    return {"cam": tuple(c + side * d for c, d in zip(cam, right)), "yaw": yaw, "pitch": pitch, "vfov": 90.0,
            "shift": -0.016 * (view - 0.5)}


# ---------------------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------------------

def _view(gbuffer):
    gb = jt.DeviceGBuffer(*gbuffer)
    return gb, torch.zeros((gb.height, gb.width, 4), dtype=torch.uint8, device=DEVICE)


def prepare(case, seed):
    return {"frame": _prepare_frame, "motion": _prepare_frame, "bake": _prepare_bake, "float": _prepare_float,
            "raster": _prepare_raster}[case["kind"]](case, seed)


def _prepare_frame(case, seed):
    gen, rng = torch.Generator(DEVICE).manual_seed(seed), random.Random(seed)
    w, h = case["width"], case["height"]
    ctx = jt.Context(0)
    sizes, nlevels = _upload_textures(ctx, case, rng, gen)
    if case["tuned"]:
        ctx.set_tuning(**{**ctx.tuning(), "decode_mcus_per_warp": 16, "decode_warps": 12, "decode_ctas_per_sm": 1})
    s = {"kind": case["kind"], "mode": case["mode"], "ctx": ctx, "filter": FILTERS[case["filter"]], "graphs": []}
    if case["kind"] == "motion":
        p = _pose(case, seed, 0)
        frames = [[_view(_scene_gbuffer(w, h, sizes, nlevels, seed, **{**p, "yaw": p["yaw"] + 6.0 * i}, quads=100))]
                  for i in range(case["directions"])]
        ctx.set_block_cache(True)
    elif case["textures"] == 1:
        frames = [[_view(_affine_gbuffer(w, h, seed + i)) for i in range(case["views"])]]
    else:
        frames = [[_view(_scene_gbuffer(w, h, sizes, nlevels, seed, **_pose(case, seed, i)))
                   for i in range(case["views"])]]
    s["frames"] = frames
    if case["mode"] == "graph":
        s["graphs"] = [ctx.frame_graph(f, s["filter"]) for f in frames]
    return s


def _prepare_bake(case, seed):
    gen = torch.Generator(DEVICE).manual_seed(seed)
    n, size = case["textures"], case["size"]
    samp = [{"420": 420, "444": 444, "mixed": 444 if t % 2 else 420}[case["sampling"]] for t in range(n)]
    ctx = jt.Context(0, max_cache_blocks=sum((-(-size // 16)) ** 2 + (32 if s == 420 else 1 + size // 8) for s in samp))
    views = []
    px, py = _pixels(size, size)
    uv = torch.stack([px / size, py / size], -1)
    for t in range(n):
        image = _noise_image(gen, size, size)
        ctx.upload(t, 0, _encode([image], case["quality"], samp[t], "standard", "standard")[0])
        tex = torch.full((size, size), t, dtype=torch.long, device=DEVICE)
        views.append(_view(_gbuffer(uv, tex, torch.zeros_like(tex))))
    return {"kind": "bake", "mode": "frame", "ctx": ctx, "filter": jt.FILTER_NEAREST, "frames": [views], "graphs": []}


def _float_inputs(case, seed):
    gen = torch.Generator(DEVICE).manual_seed(seed)
    n, size, w, h = case["textures"], case["size"], case["width"], case["height"]
    qt = _quant_tables(75)
    q = torch.tensor(np.concatenate([qt[:1].repeat(4, 0), qt[1:].repeat(2, 0)]).astype(np.float32), device=DEVICE)
    coef = torch.empty((n, size // 16, size // 16, 6, 64), dtype=torch.float32, device=DEVICE)
    for t in range(n):
        c, mx, my = _quantised(_noise_image(gen, size, size), 420, qt)
        coef[t] = (c.float() * q).reshape(my, mx, 6, 64)
    r = random.Random(seed)
    gb = _scene_gbuffer(w, h, [(size, size)] * n, [1] * n, seed, yaw=r.uniform(0, 360), pitch=r.uniform(-35, -20),
                        quads=0, mips=False)
    grad = torch.randn((h, w, 3), device=DEVICE, generator=gen)
    return coef, gb, grad


def _prepare_float(case, seed):
    coef, gb, grad = _float_inputs(case, seed)
    ctx = jt.Context(0, max_cache_blocks=case["textures"] * (case["size"] // 16) ** 2)
    ctx.register_coeff_textures(0, case["textures"], case["size"], case["size"])
    return {"kind": "float", "ctx": ctx, "coef": coef.requires_grad_(True), "gb": jt.DeviceGBuffer(*gb), "grad": grad}


# What Context.raster_scene takes for one quad.
_QUAD = np.dtype([("cx", "<f4", 4), ("cy", "<f4", 4), ("ex", "<f4", 4), ("ey", "<f4", 4), ("h", "<f4", 9),
                  ("rep", "<f4"), ("cs", "<f4"), ("sn", "<f4"), ("ou", "<f4"), ("ov", "<f4"), ("tex", "<i4"),
                  ("x0", "<i4"), ("y0", "<i4"), ("x1", "<i4"), ("y1", "<i4")])


def _scene_quad(r, width, height, ntex):
    """A convex quad of a frame 1000 units high and the projective map of it to the unit square."""
    wn = 1000.0 * width / height
    cx, cy, a0, rad = r.random() * wn, r.random() * 1000, r.uniform(0, 2 * math.pi), r.uniform(20, 90)
    ang = [a0 + i * math.pi / 2 + r.uniform(-0.12, 0.12) for i in range(4)]
    rr = [rad * r.uniform(0.85, 1.0) for _ in range(4)]
    x = np.array([cx + q * math.cos(a) for q, a in zip(rr, ang)])
    y = np.array([cy + q * math.sin(a) for q, a in zip(rr, ang)])
    rows, rhs = [], []
    for i, (s, t) in enumerate(((0, 0), (1, 0), (1, 1), (0, 1))):
        rows += [[x[i], y[i], 1, 0, 0, 0, -s * x[i], -s * y[i]], [0, 0, 0, x[i], y[i], 1, -t * x[i], -t * y[i]]]
        rhs += [s, t]
    q = np.zeros((), _QUAD)
    q["cx"], q["cy"], q["ex"], q["ey"] = x, y, np.roll(x, -1) - x, np.roll(y, -1) - y
    q["h"] = np.append(np.linalg.solve(np.array(rows, np.float64), np.array(rhs, np.float64)), 1.0)
    turn = r.uniform(0, 2 * math.pi)
    q["rep"], q["cs"], q["sn"], q["ou"], q["ov"] = r.uniform(0.5, 2), math.cos(turn), math.sin(turn), r.random(), r.random()
    q["tex"] = r.randrange(ntex)
    k = 1000.0 / height
    q["x0"], q["x1"] = max(0, int(x.min() / k) - 1), min(width - 1, int(x.max() / k) + 2)
    q["y0"], q["y1"] = max(0, int(y.min() / k) - 1), min(height - 1, int(y.max() / k) + 2)
    return q


def _prepare_raster(case, seed):
    r = random.Random(seed)
    w, h, n = case["width"], case["height"], case["textures"]
    side = [1024 << r.randrange(3) for _ in range(n)]
    th, f32 = math.tan(math.radians(30.0)), np.float32
    d = SimpleNamespace(width=w, height=h, cam=np.array([r.uniform(-5, 5), 1.7, r.uniform(-5, 5)], f32),
                        rot=_rotation(r.uniform(0, 360), r.uniform(-35, -15)).astype(f32).reshape(-1), ax=2.0 / w,
                        ay=2.0 / h, tan_x=th * w / h, tan_y=th, max_t=600.0, kx=1000.0 / h, ky=1000.0 / h, shift=0.0,
                        cell_seed=seed * 2654435761 & 0xFFFFFFFF, tex_w=np.array(side, np.int32),
                        tex_h=np.array(side, np.int32),
                        tex_levels=np.array([1 + int(math.log2(s)) for s in side], np.int32), use_mips=case["mips"],
                        quads=np.array([_scene_quad(r, w, h, n) for _ in range(case["quads"])], _QUAD))
    return {"kind": "raster", "ctx": jt.Context(0, max_cache_blocks=16), "scene": d,
            "gb": jt.DeviceGBuffer.empty(w, h, DEVICE)}


def run(state):
    ctx, kind = state["ctx"], state["kind"]
    if kind == "float":
        frame = ctx.colorize_float_autograd(state["gb"], state["coef"])
        (grad,) = torch.autograd.grad(frame, state["coef"], state["grad"])
        return {"frame": frame.detach(), "grad": grad}
    if kind == "raster":
        gb = state["gb"]
        ctx.raster_scene(state["scene"], gb)
        return {"uv": gb.uv, "tex_id": gb.tex_id, "mip": gb.mip}
    if state["mode"] == "graph":
        for g in state["graphs"]:
            ctx.graph_launch(g)
    elif state["mode"] == "frame":
        for f in state["frames"]:
            ctx.frame(f, state["filter"])
    else:
        ((gb, out),) = state["frames"][0]
        ctx.mark(gb, state["filter"])
        ctx.decode()
        ctx.colorize(gb, state["filter"], out)
    return [out for f in state["frames"] for _, out in f]


def exact(case, seed):
    """The float chain in 64 bits. The other cases return bytes and ids, and the rasteriser's uv
    is a fixed sequence of rounded fp32 operations (its cells and edges depend on them)."""
    if case["kind"] != "float":
        return None
    coef, (uv, tex_id, _), grad = _float_inputs(case, seed)
    c = coef.double().requires_grad_(True)
    n, my, mx = c.shape[:3]
    size = case["size"]
    a = _dct_matrix(torch.float64)
    f = (a.T @ c.reshape(-1, 8, 8) @ a).reshape(n, my, mx, 6, 8, 8)
    luma = f[:, :, :, :4].reshape(n, my, mx, 2, 2, 8, 8).permute(0, 1, 3, 5, 2, 4, 6).reshape(-1) + 128
    ch = f[:, :, :, 4:].permute(0, 3, 1, 4, 2, 5).reshape(n, 2, size // 2, size // 2)
    ok = tex_id >= 0
    tex = torch.where(ok, tex_id, 0).long()
    xs, ys = uv[..., 0] * float(size) - 0.5, uv[..., 1] * float(size) - 0.5  # fp32, as the path addresses
    x0, y0 = torch.floor(xs), torch.floor(ys)
    fx, fy = (xs - x0).double(), (ys - y0).double()
    out = 0.0
    for dx, dy, wt in ((0, 0, (1 - fx) * (1 - fy)), (1, 0, fx * (1 - fy)), (0, 1, (1 - fx) * fy), (1, 1, fx * fy)):
        x, y = (x0.long() + dx) % size, (y0.long() + dy) % size
        lum = luma[(tex * size + y) * size + x]
        cb, cr = ch[tex, 0, y // 2, x // 2], ch[tex, 1, y // 2, x // 2]
        rgb = torch.stack([lum + 1.402 * cr, lum - 0.344136 * cb - 0.714136 * cr, lum + 1.772 * cb], -1)
        out = out + (wt * ok)[..., None] * rgb
    (g,) = torch.autograd.grad(out, c, grad.double())
    return {"frame": out.detach(), "grad": g}
