"""Performance cases of the LATCH library: the calls a program makes, over the sizes it makes
them at.

Each case goes through the package's public entry points (``paper_1609_03986_gb300``) with
inputs drawn on the GPU from a seed: images are blurred noise with filled ellipses on top,
keypoints are uniform in the image with random orientations and scales (or upright), descriptor
sets are random with one planted near-duplicate per query.  Every output is bytes or whole
numbers (descriptors, keypoint records, match records), so two builds agree only when they are
equal and no case needs a floating-point reference.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1609_03986_gb300 as P
from paper_1609_03986_gb300 import synth

BORDER = 32              # keypoints keep this distance from the image border
SCALES = (1.0, 1.5, 2.25)
RATIO = 0.8
FAST_T = 20


def listed():
    return [
        # ---- plain calls, one image ----
        # a thumbnail or a tracked region with a few hundred keypoints: launches and latency
        {"name": "extract_region", "kind": "extract", "width": 321, "height": 243, "n": 257, "oriented": True,
         "weighted": False},
        # the upright pair workload, one image of it
        {"name": "extract_vga_upright", "kind": "extract", "width": 640, "height": 480, "n": 2000,
         "oriented": False, "weighted": False},
        # the oriented and scaled pair workload, one image of it
        {"name": "extract_hd", "kind": "extract", "width": 1920, "height": 1080, "n": 10000, "oriented": True,
         "weighted": False},
        # the same with weighted 8x8 patches
        {"name": "extract_hd_weighted", "kind": "extract", "width": 1920, "height": 1080, "n": 10000,
         "oriented": True, "weighted": True},
        # ---- plain matching, path chosen by the library ----
        # the upright pair's two descriptor sets
        {"name": "match_2k", "kind": "match", "nq": 2000, "nt": 2000, "k": 2},
        # the oriented pair's
        {"name": "match_10k", "kind": "match", "nq": 10000, "nt": 10000, "k": 2},
        # queries against a large gallery
        {"name": "match_gallery", "kind": "match", "nq": 16384, "nt": 1 << 20, "k": 2},
        # ---- keypoints found by the library: every level of the pyramid of a photograph ----
        {"name": "pyramid_photo", "kind": "pyramid", "width": 4000, "height": 3000, "levels": 3,
         "max_kps": 1 << 17},
        # ---- batched: structure from motion, every image against its next 8 ----
        {"name": "batch_sfm", "kind": "batch", "width": 4000, "height": 3000, "images": 64, "kmin": 5000,
         "kmax": 50000, "neighbours": 8},
        # the oriented pair from and to host memory
        {"name": "host_pair_hd", "kind": "host", "width": 1920, "height": 1080, "images": 2, "kmin": 10000,
         "kmax": 10000, "neighbours": 1},
        # ---- dense per-pixel descriptors of a stereo pair and their windowed matching ----
        {"name": "dense_pair_vga", "kind": "dense", "width": 640, "height": 480, "radius": 8, "k": 2},
        # ---- serving: one request from host memory against a resident gallery, waited for ----
        {"name": "serve_request", "kind": "serve", "width": 1920, "height": 1080, "n": 10000, "gallery": 100000},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo=200, hi=4000):
    """Width and height with a photograph's aspect, odd values included."""
    w = _log_int(rng, lo, hi)
    return w, max(150, int(w * rng.uniform(0.55, 0.8)))


def draw(rng):
    kind = rng.choice(["extract", "extract", "match", "match", "pyramid", "batch", "host", "dense", "serve"])
    if kind == "extract":
        w, h = _size(rng)
        return {"kind": kind, "width": w, "height": h, "n": _log_int(rng, 100, min(50000, w * h // 40)),
                "oriented": rng.random() < 0.7, "weighted": rng.random() < 0.25}
    if kind == "match":
        nq = _log_int(rng, 100, 50000)
        nt = _log_int(rng, 100, min(1 << 20, (1 << 34) // nq))
        return {"kind": kind, "nq": nq, "nt": nt, "k": rng.choice([1, 2, 2])}
    if kind == "pyramid":
        w, h = _size(rng)
        return {"kind": kind, "width": w, "height": h, "levels": rng.choice([1, 2, 3, 3]), "max_kps": 1 << 17}
    if kind in ("batch", "host"):
        w, h = _size(rng, 400, 4000 if kind == "batch" else 2000)
        kmax = min(50000 if kind == "batch" else 10000, w * h // 40)
        kmin = _log_int(rng, 200, kmax)
        return {"kind": kind, "width": w, "height": h, "images": rng.randint(2, 24 if kind == "batch" else 6),
                "kmin": kmin, "kmax": rng.randint(kmin, kmax), "neighbours": rng.randint(1, 8)}
    if kind == "dense":
        w, h = _size(rng, 200, 1200)
        return {"kind": kind, "width": w, "height": h, "radius": rng.randint(2, P_MAX_RADIUS),
                "k": rng.choice([1, 2, 2])}
    w, h = _size(rng, 400, 2000)
    return {"kind": kind, "width": w, "height": h, "n": _log_int(rng, 200, min(20000, w * h // 40)),
            "gallery": _log_int(rng, 1000, 200000)}


P_MAX_RADIUS = 16        # the largest search radius of the windowed matcher


# ---- inputs ------------------------------------------------------------------------------

def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFF)
    return g


def _image(seed, salt, w, h, n_ellipses=200):
    """(h, pitch) uint8: noise blurred by a Gaussian (sigma 1.5, radius 5), ellipses on top.  Only
    elementwise float32 steps, so that a seed gives the same bytes in every process."""
    g = _gen(seed, salt)
    r = 5
    taps = np.exp(-0.5 * (np.arange(-r, r + 1) / 1.5) ** 2)
    taps = [float(t) for t in taps / taps.sum()]
    x = torch.randint(0, 256, (h + 2 * r, w + 2 * r), generator=g, device="cuda", dtype=torch.uint8).float()
    y = torch.zeros((h + 2 * r, w), device="cuda")
    for i, t in enumerate(taps):
        y += t * x[:, i:i + w]
    z = torch.zeros((h, w), device="cuda")
    for i, t in enumerate(taps):
        z += t * y[i:i + h]
    img = z.round_().clamp_(0, 255).to(torch.uint8)
    rs = np.random.RandomState((int(seed) * 31 + salt) & 0x7FFFFFFF)
    for _ in range(n_ellipses):
        cx, cy = rs.randint(0, w), rs.randint(0, h)
        a, b = (max(2, int(min(w, h) * (0.01 + 0.09 * rs.rand()))) for _ in range(2))
        x0, x1, y0, y1 = max(0, cx - a), min(w, cx + a + 1), max(0, cy - b), min(h, cy + b + 1)
        xs = torch.arange(x0 - cx, x1 - cx, device="cuda")
        ys = torch.arange(y0 - cy, y1 - cy, device="cuda")
        inside = ((xs * xs * (b * b))[None, :] + (ys * ys * (a * a))[:, None]) <= a * a * b * b
        img[y0:y1, x0:x1].masked_fill_(inside, int(rs.randint(0, 256)))
    out = torch.zeros((h, (w + 15) // 16 * 16), dtype=torch.uint8, device="cuda")
    out[:, :w] = img
    return out


def _keypoints(seed, salt, w, h, n, oriented):
    """(n, 12) uint8 packed keypoint records."""
    g = _gen(seed, salt)

    def ints(lo, hi):
        return torch.randint(lo, hi, (n,), generator=g, device="cuda", dtype=torch.int32)

    x, y = ints(BORDER, w - BORDER), ints(BORDER, h - BORDER)
    b, s = (ints(0, 32), ints(0, len(SCALES))) if oriented else (torch.zeros_like(x), torch.zeros_like(x))
    return torch.stack([x, y, b | (s << 8)], dim=1).contiguous().view(torch.uint8).reshape(n, 12)


def _descriptors(seed, salt, n):
    return torch.randint(0, 256, (n, 64), generator=_gen(seed, salt), device="cuda", dtype=torch.uint8)


def _planted(seed, nq, nt):
    """Queries and a train set that holds a copy of each query with about 40 of its bits flipped."""
    q, t = _descriptors(seed, 1, nq), _descriptors(seed, 2, nt)
    g = _gen(seed, 3)
    m = min(nq, nt)
    slots = torch.randperm(nt, generator=g, device="cuda")[:m]
    weights = torch.tensor([1 << i for i in range(8)], device="cuda", dtype=torch.uint8)
    for i0 in range(0, m, 4096):
        i1 = min(m, i0 + 4096)
        flips = torch.rand((i1 - i0, 64, 8), generator=g, device="cuda") < 40.0 / 512.0
        t[slots[i0:i1]] = q[i0:i1] ^ (flips * weights).sum(-1).to(torch.uint8)
    return q, t


_contexts = {}


def _context(weighted=False):
    """The program's context (one per option set, kept for the life of the process)."""
    if weighted not in _contexts:
        trip = synth.triplets(lo=3, hi=43) if weighted else synth.triplets()
        ctx = P.Context(0, scales=SCALES, triplets=trip)
        if weighted:  # a Gaussian over the 8x8 patch
            d = np.arange(8) - 3.5
            P.latch_set_patch_weights(ctx.handle, np.rint(
                255 * np.exp(-(d[:, None] ** 2 + d[None, :] ** 2) / (2 * 2.0 ** 2))).astype(np.uint8))
        _contexts[weighted] = ctx
    return _contexts[weighted]


def _stream():
    return int(torch.cuda.current_stream().cuda_stream)


def _counts(case):
    """Keypoints of each image: uneven, the same for every seed (the outputs keep their shapes)."""
    rs = np.random.RandomState(case["images"] * 1000003 + case["kmin"])
    return [int(v) for v in rs.randint(case["kmin"], case["kmax"] + 1, case["images"])]


def _pinned(t):
    out = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    out.copy_(t)
    return out


def _zeros(n, width):
    return torch.zeros((n, width), dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    s, kind = dict(case), case["kind"]
    w, h = case.get("width"), case.get("height")
    if kind == "extract":
        s["ctx"] = _context(case["weighted"])
        s["img"] = _image(seed, 10, w, h)
        s["kps"] = _keypoints(seed, 11, w, h, case["n"], case["oriented"])
        s["out"] = _zeros(case["n"], 64)
    elif kind == "match":
        s["ctx"] = _context()
        s["q"], s["t"] = _planted(seed, case["nq"], case["nt"])
        s["out"] = _zeros(case["nq"], 16)
    elif kind == "pyramid":
        s["ctx"] = _context()
        s["img"] = _image(seed, 10, w, h)
        s["kps"], s["desc"] = _zeros(case["max_kps"], 12), _zeros(case["max_kps"], 64)
        s["count"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    elif kind in ("batch", "host"):
        s["ctx"] = _context()
        n = _counts(case)
        imgs = [_image(seed, 100 + 2 * i, w, h) for i in range(case["images"])]
        kps = torch.cat([_keypoints(seed, 101 + 2 * i, w, h, c, True) for i, c in enumerate(n)])
        pairs = synth.batch_pairs(case["images"], case["neighbours"])
        matches = sum(n[a] for a, _ in pairs)
        if kind == "batch":
            s["imgs"], s["kps"] = imgs, kps
            s["desc"], s["out"] = _zeros(sum(n), 64), _zeros(matches, 16)
            make = P.BatchDesc
        else:
            s["imgs"], s["kps"] = [_pinned(i) for i in imgs], _pinned(kps)
            s["desc"] = torch.zeros((sum(n), 64), dtype=torch.uint8).pin_memory()
            s["out"] = torch.zeros((matches, 16), dtype=torch.uint8).pin_memory()
            make = P.HostBatchDesc
        s["batch"] = make([(i, w, h, i.stride(0)) for i in s["imgs"]], n, s["kps"], s["desc"], pairs, 2, RATIO,
                          s["out"])
    elif kind == "dense":
        s["ctx"] = _context()
        base = _image(seed, 10, w + 8, h + 8)  # the second view is the first moved by (3, -2)
        s["img"] = [torch.zeros((h, (w + 15) // 16 * 16), dtype=torch.uint8, device="cuda") for _ in range(2)]
        s["img"][0][:, :w] = base[4:4 + h, 4:4 + w]
        s["img"][1][:, :w] = base[6:6 + h, 1:1 + w]
        s["desc"] = [_zeros(w * h, 64) for _ in range(2)]
        s["out"] = _zeros(w * h, 16)
    elif kind == "serve":
        s["session"] = P.Session(synth.triplets(), hbm_budget=1 << 30, max_gallery_rows=1 << 18, max_batch=16,
                                 max_batch_kps=1 << 16)
        s["img"] = _pinned(_image(seed, 10, w, h)).numpy()
        s["kps"] = _pinned(_keypoints(seed, 11, w, h, case["n"], True)).numpy()
        s["gallery_id"] = s["session"].add_gallery(_descriptors(seed, 12, case["gallery"]).cpu().numpy())
    return s


def run(s):
    kind = s["kind"]
    w, h = s.get("width"), s.get("height")
    if kind == "extract":
        return s["ctx"].extract(s["img"], w, h, s["kps"], out=s["out"])
    if kind == "match":
        return s["ctx"].match(s["q"], s["t"], s["k"], RATIO, out=s["out"])
    if kind == "pyramid":
        P.latch_detect_pyramid(s["ctx"].handle, s["img"], w, h, s["img"].stride(0), FAST_T, s["levels"],
                               s["max_kps"], s["kps"], s["count"], s["desc"], _stream())
        return {"kps": s["kps"], "count": s["count"], "desc": s["desc"]}
    if kind == "batch":
        P.latch_batch_run(s["ctx"].handle, s["batch"], _stream())
        return {"desc": s["desc"], "matches": s["out"]}
    if kind == "host":
        P.latch_batch_run_host(s["ctx"].handle, s["batch"], _stream())
        return {"desc": s["desc"], "matches": s["out"]}
    if kind == "dense":
        a, b = (s["ctx"].dense_extract(s["img"][i], w, h, out=s["desc"][i]) for i in range(2))
        m = s["ctx"].dense_match(a, b, w, h, s["radius"], s["k"], RATIO, out=s["out"])
        return {"a": a, "b": b, "matches": m}
    ticket = s["session"].submit(s["img"], w, h, s["kps"], s["gallery_id"], 2, RATIO, want_desc=True)
    _, matches, desc = s["session"].wait(ticket)
    return {"desc": desc, "matches": matches.view(np.uint8).reshape(-1, 16)}


# ---- work of one pass --------------------------------------------------------------------

_DESC_OPS = 512 * 2 * 49 * 2      # Eq. 1: two 7x7 sums of squared differences per bit
_WEIGHTED_OPS = 512 * 2 * 64 * 3  # with 8x8 weighted patches
_PAIR_OPS = 2 * 512               # one 512-bit distance as a dot product
_DENSE_OPS = 512 * 9              # per pixel: product image and separable box sum


def work(case):
    kind = case["kind"]
    w, h = case.get("width", 0), case.get("height", 0)
    if kind == "extract":
        ops = _WEIGHTED_OPS if case["weighted"] else _DESC_OPS
        return {"bytes": w * h + case["n"] * (12 + 64), "flops": case["n"] * ops}
    if kind == "match":
        return {"bytes": 64 * (case["nq"] + case["nt"]) + 16 * case["nq"], "flops": _PAIR_OPS * case["nq"] * case["nt"]}
    if kind == "pyramid":  # about one keypoint per 280 pixels of a photograph's levels
        px = sum(int(w / s) * int(h / s) for s in SCALES[:case["levels"]])
        n = min(case["max_kps"], px // 280)
        return {"bytes": w * h + n * (12 + 64), "flops": 30 * px + n * _DESC_OPS}
    if kind in ("batch", "host"):
        k = _counts(case)
        pairs = synth.batch_pairs(case["images"], case["neighbours"])
        return {"bytes": case["images"] * w * h + sum(k) * (12 + 64) + sum(k[a] for a, _ in pairs) * 16,
                "flops": sum(k) * _DESC_OPS + sum(k[a] * k[b] for a, b in pairs) * _PAIR_OPS}
    if kind == "dense":
        side = 2 * case["radius"] + 1
        return {"bytes": 2 * w * h * (1 + 64) + w * h * (128 + 16),
                "flops": 2 * w * h * _DENSE_OPS + w * h * side * side * _PAIR_OPS}
    n = case["n"]
    return {"bytes": w * h + n * (12 + 64 + 16) + case["gallery"] * 64,
            "flops": n * _DESC_OPS + n * case["gallery"] * _PAIR_OPS}
