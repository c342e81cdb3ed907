"""Measured cases: what a user of this package has it do, each through the
public entry points, with seeded synthetic inputs made on the GPU.

The kinds, and what each stands for in real use:

* ``pair``     one small image pair from pixels to offsets: CFOG of both images
               and one `cfog_match` launch with a handful of control points
               (CPs) -- the smallest whole call, where latency counts.
* ``step``     the whole batched step: CFOG of both images, block-based Harris
               CPs, one batched launch over CPs of uneven template side N and
               search radius r.
* ``match``    matching alone on features that are already resident: the
               map-like pair (one class N 96, r 20) in FP32 and in BF16, one
               2048-row band of a 20000-pixel-wide 12-bit scene with a
               georeferenced search prior per CP, and a served batch of CPs
               of several jobs of different image sizes.
* ``extract``  CFOG alone: the benchmark's image, a large 12-bit image with
               ragged sides, and (drawn) the other channel counts, Gaussian
               radii and the binned orientation scheme.
* ``detect``   Harris CPs of a large 12-bit image with scene-sized cells.
* ``fhog``     the 36-channel pixel-wise HOG of both images and matching on it.
* ``reject``   iterative outlier rejection of a scene's CPs.
* ``rectify``  piecewise-linear rectification of a large 12-bit image.

Sizes are those of the package's benchmark, tests and serving stream; `draw`
spreads them over the same ranges, odd sizes included.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1808_06194_gb300 as P

FP32, BF16 = 0, 1
AUTO, PAIR_TMEM = 0, 4
EQ2, BINS = 0, 1
MIX = "48/64/96/128"      # template sides of the batched step


def listed():
    return [
        # one 256 x 256 pair, one 64 x 64 template at the centre, radius 16
        {"name": "pair_256", "kind": "pair", "size": 256, "grid": 1, "tmpl": "64", "r_lo": 16, "r_hi": 16},
        # the benchmark's step: 1024 Harris CPs, N in {48..128}, r in 8..20, in
        # the variant the autotuner picks for this mix on this GPU
        {"name": "step_2048", "kind": "step", "size": 2048, "grid": 32, "tmpl": MIX, "r_lo": 8, "r_hi": 20,
         "variant": PAIR_TMEM},
        # the precision workload, FP32 FFT and BF16 tensor cores: 4096 CPs
        {"name": "match_map_fp32", "kind": "match", "render": "map", "jobs": 1, "h": 4096, "w": 4096, "cps": 4096,
         "tmpl": "96", "r_lo": 20, "r_hi": 20, "prior": False, "precision": FP32, "variant": AUTO},
        {"name": "match_map_bf16", "kind": "match", "render": "map", "jobs": 1, "h": 4096, "w": 4096, "cps": 4096,
         "tmpl": "96", "r_lo": 20, "r_hi": 20, "prior": False, "precision": BF16, "variant": AUTO},
        # one band of the large scene: 1000 CPs with a search prior, one class
        {"name": "match_scene_band", "kind": "match", "render": "sar", "jobs": 1, "h": 2304, "w": 20000,
         "cps": 1000, "tmpl": "96", "r_lo": 16, "r_hi": 16, "prior": True, "precision": FP32, "variant": AUTO},
        # a served batch: CPs of ten jobs (sides 512 to 2048, one CP per
        # 64 x 64 block) in one launch
        {"name": "match_served", "kind": "match", "render": "speckle", "jobs": 10, "h": 512, "w": 2048, "cps": 0,
         "tmpl": "64/96", "r_lo": 10, "r_hi": 20, "prior": False, "precision": FP32, "variant": PAIR_TMEM},
        # CFOG of the benchmark's image, and of a large ragged 12-bit image
        {"name": "extract_2048", "kind": "extract", "h": 2048, "w": 2048, "dtype": "f32", "m": 9, "radius": 3,
         "orient": EQ2},
        {"name": "extract_8k_u16", "kind": "extract", "h": 8190, "w": 8001, "dtype": "u16", "m": 9, "radius": 3,
         "orient": EQ2},
        # Harris CPs with the large scene's cells (about 197 px a side)
        {"name": "detect_8k_u16", "kind": "detect", "h": 8192, "w": 8192, "dtype": "u16", "gy": 41, "gx": 41,
         "k": 1, "chip": 0, "margin": 80},
        # the HOG descriptor through the matcher
        {"name": "fhog_1024", "kind": "fhog", "size": 1024, "grid": 16, "tmpl": MIX, "r_lo": 8, "r_hi": 20,
         "cell": 8, "variant": AUTO},
        # the large scene's outlier rejection and rectification
        {"name": "reject_10000", "kind": "reject", "n": 10000, "outliers": 0.05, "degree": 3, "rmse": 0.3},
        {"name": "rectify_8k_u16", "kind": "rectify", "h": 8192, "w": 8192, "dtype": "u16", "grid": 41},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pair", "step", "match", "match", "match", "extract", "extract", "detect", "fhog",
                       "reject", "rectify"])
    r_lo = rng.randint(4, 24)
    r_hi = rng.randint(r_lo, min(32, r_lo + 12))
    tmpl = rng.choice([MIX, "64/96", str(rng.randint(16, 128)), "%d/%d" % (rng.randint(16, 80), rng.randint(81, 192))])
    if kind == "pair":
        return {"kind": "pair", "size": rng.randint(256, 700), "grid": rng.randint(1, 4),
                "tmpl": str(rng.randint(16, 128)), "r_lo": r_lo, "r_hi": r_lo}
    if kind == "step":
        size = _log(rng, 700, 2200)
        return {"kind": "step", "size": size, "grid": rng.randint(3, size // 64), "tmpl": tmpl, "r_lo": r_lo,
                "r_hi": r_hi, "variant": rng.choice([AUTO, PAIR_TMEM])}
    if kind == "match":
        bf16 = rng.random() < 0.3
        return {"kind": "match", "render": rng.choice(["map", "speckle", "sar"]), "jobs": 1,
                "h": rng.randint(700, 4096), "w": rng.randint(700, 6000), "cps": _log(rng, 20, 2500),
                "tmpl": str(rng.randint(16, 128)) if bf16 else tmpl, "r_lo": r_lo, "r_hi": r_hi,
                "prior": rng.random() < 0.5, "precision": BF16 if bf16 else FP32,
                "variant": AUTO if bf16 else rng.choice([AUTO, PAIR_TMEM])}
    if kind == "extract":
        orient = rng.choice([EQ2, EQ2, BINS])
        return {"kind": "extract", "h": _log(rng, 61, 6000), "w": _log(rng, 67, 6000), "dtype": rng.choice(["f32", "u16"]),
                "m": rng.choice([6, 8, 9, 9, 12]), "radius": 3 if orient == BINS else rng.choice([2, 3, 3, 4]),
                "orient": orient}
    if kind == "detect":
        h, w = _log(rng, 300, 8192), _log(rng, 300, 8192)
        return {"kind": "detect", "h": h, "w": w, "dtype": rng.choice(["f32", "u16"]), "gy": max(2, h // rng.randint(64, 200)),
                "gx": max(2, w // rng.randint(64, 200)), "k": rng.choice([1, 1, 2, 4]), "chip": rng.choice([0, 0, 60]),
                "margin": rng.randint(0, 100)}
    if kind == "fhog":
        size = rng.randint(500, 1100)
        return {"kind": "fhog", "size": size, "grid": rng.randint(2, 12), "tmpl": str(rng.randint(16, 100)), "r_lo": r_lo,
                "r_hi": r_hi, "cell": rng.choice([4, 8]), "variant": AUTO}
    if kind == "reject":
        return {"kind": "reject", "n": _log(rng, 300, 10000), "outliers": rng.choice([0.02, 0.05]), "degree": rng.choice([1, 2, 3]),
                "rmse": 0.3}
    return {"kind": "rectify", "h": _log(rng, 500, 8000), "w": _log(rng, 500, 8000), "dtype": rng.choice(["f32", "u16"]),
            "grid": rng.randint(4, 41)}


# ---------------------------------------------------------------- inputs --

DEV = "cuda"


def _gen(seed, salt=0):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 1000003 + salt)


def _rand(g, *shape):
    return torch.rand(shape, generator=g, device=DEV)


def _sides(case):
    return [int(v) for v in case["tmpl"].split("/")]


def _texture(g, h, w):
    """Random rectangles (40 per 256 x 256, sides 8..64) plus blurred white noise, in [0, 255]."""
    n = max(1, round(40 * h * w / 65536))
    y0, x0 = (_rand(g, n) * h).long(), (_rand(g, n) * w).long()
    y1 = torch.minimum(y0 + 8 + (_rand(g, n) * 57).long(), torch.tensor(h, device=DEV))
    x1 = torch.minimum(x0 + 8 + (_rand(g, n) * 57).long(), torch.tensor(w, device=DEV))
    val = (_rand(g, n) * 256).int()
    acc = torch.zeros((h + 1) * (w + 1), dtype=torch.int32, device=DEV)   # integers: any order of the sums
    for y, x, s in ((y0, x0, 1), (y1, x0, -1), (y0, x1, -1), (y1, x1, 1)):
        acc.index_add_(0, y * (w + 1) + x, s * val)
    img = acc.view(h + 1, w + 1).cumsum(0, dtype=torch.int32).cumsum(1, dtype=torch.int32)[:h, :w].float()
    noise = torch.randn((h, w), generator=g, device=DEV) * 20.0
    taps = [math.exp(-t * t / 4.5) for t in range(-5, 6)]
    for axis in (0, 1):
        noise = sum(c / sum(taps) * torch.roll(noise, t, axis) for t, c in zip(range(-5, 6), taps))
    img += noise
    img -= img.min()
    return img * (255.0 / img.max().clamp(min=1e-6))


def _speckle(g, shape):
    """Gamma(4, 1/4): the mean of four unit exponentials."""
    s = torch.zeros(shape, device=DEV)
    for _ in range(4):
        s -= torch.log(torch.rand(shape, generator=g, device=DEV).clamp(min=1e-7))
    return s * 0.25


def _warp(img, dy, dx):
    """Bilinear sample of img at (y - dy, x - dx), borders repeated."""
    h, w = img.shape
    ys = torch.arange(h, device=DEV, dtype=torch.float32)[:, None] - dy
    xs = torch.arange(w, device=DEV, dtype=torch.float32)[None, :] - dx
    ys, xs = ys.clamp(0, h - 1).expand(h, w), xs.clamp(0, w - 1).expand(h, w)
    yi, xi = ys.floor().clamp(max=h - 2).long(), xs.floor().clamp(max=w - 2).long()
    fy, fx = ys - yi, xs - xi
    flat = img.reshape(-1)
    at = yi * w + xi
    top = flat[at] * (1 - fx) + flat[at + 1] * fx
    return top * (1 - fy) + (flat[at + w] * (1 - fx) + flat[at + w + 1] * fx) * fy


def _pair(seed, h, w, render):
    """Reference and sensed image and the displacement (dy, dx) tensors of the pair."""
    g = _gen(seed)
    A = _texture(g, h, w)
    p = _rand(g, 10).tolist()
    sy, sx = int(p[0] * 13) - 6, int(p[1] * 13) - 6
    Y = torch.arange(h, device=DEV, dtype=torch.float32)[:, None]
    X = torch.arange(w, device=DEV, dtype=torch.float32)[None, :]
    if render == "shift":
        dy = torch.full((1, 1), float(sy), device=DEV)
        dx = torch.full((1, 1), float(sx), device=DEV)
    elif render == "sar":     # shift and a 0.1 degree rotation about the centre
        th = math.radians(0.1)
        dy = sy + th * (X - w / 2) + 0 * Y
        dx = sx - th * (Y - h / 2) + 0 * X
    else:                     # shift and low-frequency sines
        dy = sy + 3 * torch.sin(2 * math.pi * (p[2] * X / w + p[3] * Y / h + p[4]))
        dx = sx + 3 * torch.sin(2 * math.pi * (p[5] * X / w + p[6] * Y / h + p[7]))
    if render == "map":       # six levels, 1-px boundary lines, N(0, 10^2)
        lab = (A / 255.0 * 6).clamp(max=5.999).floor()
        B = (lab + 0.5) * (255.0 / 6)
        edge = torch.zeros_like(B, dtype=torch.bool)
        edge[:, :-1] |= lab[:, :-1] != lab[:, 1:]
        edge[:-1] |= lab[:-1] != lab[1:]
        B = torch.where(edge, torch.zeros_like(B), B) + 10.0 * torch.randn((h, w), generator=g, device=DEV)
    elif render == "sar":     # 12-bit log-speckled remap
        A = (A * 16.0).round()
        B = torch.log1p(A * _speckle(g, (h, w))) * (4095.0 / math.log1p(4095.0 * 4.0))
    else:
        B = 255.0 * (1.0 - (A / 255.0).sqrt()) * _speckle(g, (h, w))
    B = _warp(B, dy, dx)
    if render == "sar":
        return A.clamp(0, 4095).int().to(torch.uint16), B.round().clamp(0, 4095).int().to(torch.uint16), dy, dx
    return A.contiguous(), B.contiguous(), dy, dx


def _image(seed, h, w, dtype):
    img = _texture(_gen(seed), h, w)
    return (img * 16.0).round().clamp(0, 4095).int().to(torch.uint16) if dtype == "u16" else img.contiguous()


def _class_rows(case, seed, n):
    """Per-CP template side and radius (int32, on the device)."""
    g = _gen(seed, 77)
    s = torch.tensor(_sides(case), device=DEV, dtype=torch.int32)
    tm = s[(_rand(g, n) * len(s)).long().clamp(max=len(s) - 1)]
    rd = case["r_lo"] + (_rand(g, n) * (case["r_hi"] - case["r_lo"] + 1)).int().clamp(max=case["r_hi"] - case["r_lo"])
    return tm.contiguous(), rd.int().contiguous()


def _margin(case, extra=16):
    return max(_sides(case)) // 2 + case["r_hi"] + extra


def _served_sides(case):
    """Sides of the jobs: log-spaced, rounded to 16."""
    k = case["jobs"]
    return [int(math.exp(math.log(case["h"]) + (math.log(case["w"]) - math.log(case["h"])) * i / max(1, k - 1))) // 16 * 16
            for i in range(k)]


def _match_images(case, seed):
    """The pairs of a match case, with every CP: [(A, B, dy, dx)], cps, job of CP, prior (or None)."""
    m = _margin(case, 24)
    if case["jobs"] > 1:
        pairs, cps, job = [], [], []
        for j, s in enumerate(_served_sides(case)):
            pairs.append(_pair(seed * 64 + j, s, s, case["render"]))
            n = max(1, (s - 2 * m) // 64)
            c = m + 32 + 64 * torch.arange(n, device=DEV)
            off = (_rand(_gen(seed, 500 + j), n, n, 2) * 33).int() - 16
            cps.append(torch.stack([c[None, :] + off[..., 0], c[:, None] + off[..., 1]], -1).reshape(-1, 2).int())
            job.append(torch.full((n * n,), j, dtype=torch.int32, device=DEV))
        return pairs, torch.cat(cps).contiguous(), torch.cat(job).contiguous(), None
    A, B, dy, dx = _pair(seed, case["h"], case["w"], case["render"])
    g = _gen(seed, 5)
    h, w, n = case["h"], case["w"], case["cps"]
    m = min(m + (int(0.00175 * max(h, w) / 2) + 4 if case["render"] == "sar" else 0), min(h, w) // 2 - 8)
    cps = torch.stack([m + (_rand(g, n) * (w - 2 * m)).int(), m + (_rand(g, n) * (h - 2 * m)).int()], 1).int().contiguous()
    prior = None
    if case["prior"]:         # the true displacement, rounded, with up to 3 px of error
        y, x = cps[:, 1].long(), cps[:, 0].long()
        q = torch.stack([dx.expand(h, w)[y, x], dy.expand(h, w)[y, x]], 1).round()
        prior = (q.int() + (_rand(g, n, 2) * 7).int().clamp(max=6) - 3).int().contiguous()
    return [(A, B, dy, dx)], cps, None, prior


def _cubic(g, n, size):
    xy = (size / 16 + _rand(g, n, 2) * (size * 7 / 8)).int()
    u, v = (xy.double() / size * 2 - 1).unbind(1)
    mon = torch.stack([torch.ones_like(u), u, v, u * u, u * v, v * v, u ** 3, u * u * v, u * v * v, v ** 3])
    c = torch.randn((2, 10), generator=g, device=DEV, dtype=torch.float64) * 6.0
    return xy.contiguous(), (c[:, :, None] * mon).sum(1)


def _result_rows(d, status=None):
    """(n, 6) int32 cfog_match_result rows of offsets d (2, n)."""
    n = d.shape[1]
    res = torch.zeros((n, 6), dtype=torch.int32, device=DEV)
    f = d.float().t().contiguous()
    res[:, 0:2] = f.round().int()
    res[:, 2:4] = f.view(torch.int32)
    if status is not None:
        res[:, 5] = status
    return res.contiguous()


def _reject_inputs(case, seed):
    g = _gen(seed)
    n = case["n"]
    cps, d = _cubic(g, n, 20000)
    d = d + torch.tensor([[7.0], [-4.0]], device=DEV, dtype=torch.float64)
    if case["degree"] < 3:    # smooth data of the model's own degree
        u, v = (cps.double() / 10000 - 1).unbind(1)
        d = torch.stack([7 + 3 * u - 2 * v, -4 + u + 5 * v])
    d = d + 0.15 * torch.randn((2, n), generator=g, device=DEV, dtype=torch.float64)
    k = int(round(case["outliers"] * n))
    perm = torch.randperm(n, generator=g, device=DEV)
    out, bad = perm[:k], perm[k:k + n // 50]
    mag = 6.0 + 1.5 * torch.randperm(k, generator=g, device=DEV).double()   # distinct: no near ties
    ang = 2 * math.pi * torch.rand(k, generator=g, device=DEV, dtype=torch.float64)
    d[:, out] += torch.stack([mag * torch.cos(ang), mag * torch.sin(ang)])
    status = torch.zeros(n, dtype=torch.int32, device=DEV)
    status[bad] = 2
    return cps, _result_rows(d, status)


def _rectify_inputs(case, seed):
    g = _gen(seed, 9)
    h, w, k = case["h"], case["w"], case["grid"]
    img = _image(seed, h, w, case["dtype"])
    cy, cx = (h - 80) / k, (w - 80) / k
    j = torch.arange(k, device=DEV)
    jit = (_rand(g, k, k, 2) - 0.5) * 0.6
    y = 40 + (j[:, None] + 0.5 + jit[..., 0]) * cy
    x = 40 + (j[None, :] + 0.5 + jit[..., 1]) * cx
    cps = torch.stack([x, y], -1).reshape(-1, 2).int().contiguous()
    u, v = cps[:, 0].double() / w, cps[:, 1].double() / h
    d = torch.stack([5 + 3 * torch.sin(5 * u) + 2 * v, -3 + 4 * torch.cos(4 * v) - u])
    d = d + 0.2 * torch.randn(d.shape, generator=g, device=DEV, dtype=torch.float64)
    return img, cps, _result_rows(d)


# ------------------------------------------------------ prepare and run ----

def _features(img):
    return P.cfog_extract(img)


def prepare(case, seed):
    k = case["kind"]
    if k in ("pair", "step", "fhog"):
        s = case["size"]
        A, B, _, _ = _pair(seed, s, s, "shift" if k == "pair" else "speckle")
        n = case["grid"] ** 2
        tm, rd = _class_rows(case, seed, n)
        m = 36 if k == "fhog" else 9
        fa, fb = P.alloc_features(s, s, m), P.alloc_features(s, s, m)
        st = {"case": case, "A": A, "B": B, "tm": tm, "rd": rd, "fa": fa, "fb": fb,
              "tmax": max(_sides(case)), "rmax": case["r_hi"], "margin": _margin(case)}
        if k == "pair":
            st["cps"] = _grid_cps(case)
        else:
            st["jobs"] = P.job_table([(fa, fb)])
            st["ws"] = P.match_workspace(n)
        return st
    if k == "match":
        pairs, cps, job, prior = _match_images(case, seed)
        feats = [(_features(A), _features(B)) for A, B, _, _ in pairs]
        n = cps.shape[0]
        tm, rd = _class_rows(case, seed, n)
        return {"case": case, "feats": feats, "jobs": P.job_table(feats), "cps": cps, "job": job, "prior": prior,
                "tm": tm, "rd": rd, "tmax": max(_sides(case)), "rmax": case["r_hi"], "ws": P.match_workspace(n)}
    if k == "extract":
        img = _image(seed, case["h"], case["w"], case["dtype"])
        return {"case": case, "img": img, "p": P.params(m=case["m"], gauss_radius=case["radius"], orientation=case["orient"]),
                "out": P.alloc_features(case["h"], case["w"], case["m"])}
    if k == "detect":
        return {"case": case, "img": _image(seed, case["h"], case["w"], case["dtype"])}
    if k == "reject":
        cps, res = _reject_inputs(case, seed)
        return {"case": case, "cps": cps, "res": res, "ws": P.reject_workspace(case["n"], 1)}
    img, cps, res = _rectify_inputs(case, seed)
    tris = torch.from_numpy(P.tin_delaunay(cps)).to(DEV)
    return {"case": case, "img": img, "cps": cps, "res": res, "tris": tris,
            "ws": P.tin_workspace(tris.shape[0], case["h"], case["w"]),
            "out": torch.empty((case["h"], case["w"]), dtype=torch.float32, device=DEV)}


def _grid_cps(case):
    """CPs of a small pair: the centres of a grid over the interior."""
    m, s, k = _margin(case), case["size"], case["grid"]
    m = min(m, s // 2)
    c = [m + (s - 2 * m) * (2 * i + 1) // (2 * k) for i in range(k)]
    return torch.tensor([[x, y] for y in c for x in c], dtype=torch.int32, device=DEV)


def _matches(cps, res):
    """What a caller takes from the result rows: integer offsets and status, the SSD, and the matched points
    p + d in the sensed image (what the mapping models are fitted to), pixels."""
    f = P.unpack_results(res)
    return {"dx": f["dx"], "dy": f["dy"], "status": f["status"], "ssd": f["ssd"],
            "points": torch.add(cps, res.view(torch.float32)[:, 2:4])}


def run(st):
    case = st["case"]
    k = case["kind"]
    if k == "pair":
        P.cfog_extract(st["A"], out=st["fa"])
        P.cfog_extract(st["B"], out=st["fb"])
        res = P.cfog_match(st["fa"], st["fb"], st["cps"], st["tm"], st["rd"], st["tmax"], st["rmax"])
        return {"match": _matches(st["cps"], res), "ref": st["fa"].volume(), "sen": st["fb"].volume()}
    if k in ("step", "fhog"):
        if k == "step":
            P.cfog_extract(st["A"], out=st["fa"])
            P.cfog_extract(st["B"], out=st["fb"])
        else:
            P.cfog_extract_fhog(st["A"], cell=case["cell"], out=st["fa"])
            P.cfog_extract_fhog(st["B"], cell=case["cell"], out=st["fb"])
        g = case["grid"]
        cps = P.cfog_detect_cps(st["A"], g, g, 1, 0, st["margin"])
        res = P.cfog_match_batched(st["jobs"], 1, cps, st["tm"], st["rd"], st["tmax"], st["rmax"], m=st["fa"].m,
                                   variant=case["variant"], workspace=st["ws"])
        out = {"cps": cps, "match": _matches(cps, res)}
        if k == "fhog":
            out["ref"], out["sen"] = st["fa"].volume(), st["fb"].volume()
        return out
    if k == "match":
        res = P.cfog_match_batched(st["jobs"], case["jobs"], st["cps"], st["tm"], st["rd"], st["tmax"], st["rmax"],
                                   job_of_cp=st["job"], prior=st["prior"], precision=case["precision"],
                                   variant=case["variant"], workspace=st["ws"])
        return {"match": _matches(st["cps"], res)}
    if k == "extract":
        f = P.cfog_extract(st["img"], st["p"], out=st["out"])
        return {"volume": f.volume(), "sqnorm": f.sq()}
    if k == "detect":
        return {"cps": P.cfog_detect_cps(st["img"], case["gx"], case["gy"], case["k"], case["chip"], case["margin"])}
    if k == "reject":
        keep, order, models = P.cfog_reject_outliers(st["cps"], st["res"], None, case["degree"], case["rmse"],
                                                     workspace=st["ws"])
        # cfog_poly_model: six int32, then rmse, cx, cy, scale, coef_x[10], coef_y[10]
        return {"keep": keep, "order": order, "counts": models.view(torch.int32)[:, :6],
                "model": models.view(torch.float64)[:, 3:]}
    return {"image": P.cfog_tin_rectify(st["img"], st["cps"], st["res"], st["tris"], case["h"], case["w"],
                                        out=st["out"], workspace=st["ws"])}


# ----------------------------------------------------------------- work ----

def _match_work(case, n, m, px):
    """Feature bytes the CPs read (at most every volume once) and FFT flops, over the class draws."""
    by = fl = 0.0
    cls = [(N, r) for N in _sides(case) for r in range(case["r_lo"], case["r_hi"] + 1)]
    for N, r in cls:
        W = N + 2 * r
        by += 4.0 * m * (N * N + W * W) / len(cls)
        fl += (2 * m + 1) * 2.5 * W * W * 2 * math.log2(W) / len(cls)
    return min(n * by, 2 * 4.0 * m * px) + 24.0 * n, n * fl


def work(case):
    k = case["kind"]
    if k in ("pair", "step", "fhog"):
        px, n = case["size"] ** 2, case["grid"] ** 2
        m = 36 if k == "fhog" else 9
        b, f = _match_work(case, n, m, px)
        return {"bytes": b + 2 * px * (8 + 4 * m), "flops": f + 2 * px * m * (36 if k != "fhog" else 80)}
    if k == "match":
        if case["jobs"] > 1:
            sides, m = _served_sides(case), _margin(case, 24)
            n, px = sum(max(1, (s - 2 * m) // 64) ** 2 for s in sides), sum(s * s for s in sides)
        else:
            n, px = case["cps"], case["h"] * case["w"]
        b, f = _match_work(case, n, 9, px)
        if case["precision"] == BF16:   # the direct correlation's products
            cls = [(N, r) for N in _sides(case) for r in range(case["r_lo"], case["r_hi"] + 1)]
            f = n * sum(2.0 * 9 * N * N * (2 * r + 1) ** 2 for N, r in cls) / len(cls)
        return {"bytes": b, "flops": f}
    px = float(case["h"] * case["w"]) if "h" in case else 0.0
    isz = 2 if case.get("dtype") == "u16" else 4
    if k == "extract":
        return {"bytes": px * (isz + 4 * case["m"] + 4), "flops": px * case["m"] * (12 + 8 * case["radius"])}
    if k == "detect":
        return {"bytes": px * isz, "flops": px * 65}
    if k == "reject":
        n = case["n"]
        return {"bytes": n * 37.0, "flops": n * case["outliers"] * n * 50.0}
    return {"bytes": px * (isz + 4), "flops": px * 20}


# ----------------------------------------------------- 64-bit references ---

def _shift(a, d, axis):
    """a at index + d along axis, edge values repeated."""
    n = a.shape[axis]
    return a.index_select(axis, (torch.arange(n, device=a.device) + d).clamp(0, n - 1))


def _gradients(img):
    img = img.to(torch.float64)
    return _shift(img, 1, 1) - _shift(img, -1, 1), _shift(img, 1, 0) - _shift(img, -1, 0)


def _bins(gx, gy, m, k):
    """Magnitude share of orientation bin k: linear between the two nearest bins."""
    mag = torch.sqrt(gx * gx + gy * gy)
    t = torch.atan2(gy, gx)
    t = torch.where(t < 0, t + math.pi, t) * (m / math.pi)
    t = torch.where(t >= m, t - m, t)
    d = (t - k).abs()
    return (1 - torch.minimum(d, m - d)).clamp(min=0) * mag


def _blur(a, taps):
    R = len(taps) // 2
    for axis in (1, 0):
        a = sum(c * _shift(a, t, axis) for t, c in zip(range(-R, R + 1), taps))
    return a


def _gauss(sigma, R):
    t = [math.exp(-i * i / (2 * sigma * sigma)) for i in range(-R, R + 1)]
    return [v / sum(t) for v in t]


def _cfog64(img, m=9, R=3, orient=EQ2, sigma=float(np.float32(0.8)), eps=float(np.float32(1e-6))):
    gx, gy = _gradients(img)
    taps = _gauss(sigma, R)
    h = torch.empty((m,) + tuple(img.shape), dtype=torch.float64, device=img.device)
    for k in range(m):
        th = k * math.pi / m
        h[k] = _blur(_bins(gx, gy, m, k) if orient == BINS else (math.cos(th) * gx + math.sin(th) * gy).abs(), taps)
    z = torch.empty_like(h)
    for k in range(m):
        z[k] = (h[k - 1] + 2 * h[k] + h[(k + 1) % m]) / 4
    del h
    nrm = torch.zeros_like(gx)
    for k in range(m):
        nrm += z[k] * z[k]
    return z.div_(nrm.sqrt() + eps)


def _fhog64(img, C, eps=float(np.float32(1e-6))):
    gx, gy = _gradients(img)
    wgt = [[max(0.0, 1 - abs(d - c) / C) for d in range(-C, C + 1)] for c in (-C / 2, C / 2)]
    out = torch.empty((36,) + tuple(img.shape), dtype=torch.float64, device=img.device)
    for k in range(9):
        a = _bins(gx, gy, 9, k)
        for cx in range(2):
            ax = sum(w * _shift(a, d, 1) for d, w in zip(range(-C, C + 1), wgt[cx]) if w)
            for cy in range(2):
                out[(cy * 2 + cx) * 9 + k] = sum(w * _shift(ax, d, 0) for d, w in zip(range(-C, C + 1), wgt[cy]) if w)
    return out.div_((out * out).sum(0).sqrt() + eps)


def _harris64(img, g, margin):
    gx, gy = _gradients(img)
    taps = _gauss(1.5, 4)
    a, b, c = _blur(gx * gx, taps), _blur(gy * gy, taps), _blur(gx * gy, taps)
    resp = (a * b - c * c) - 0.04 * (a + b) ** 2
    h, w = img.shape
    ih, iw = h - 2 * margin, w - 2 * margin
    out = []
    for j in range(g):
        for i in range(g):
            y0, y1 = margin + j * ih // g, margin + (j + 1) * ih // g
            x0, x1 = margin + i * iw // g, margin + (i + 1) * iw // g
            cell = resp[y0:y1, x0:x1].reshape(-1)
            at = torch.argmax(cell)
            out.append(torch.stack([x0 + at % (x1 - x0), y0 + at // (x1 - x0)]))
    return torch.stack(out)


def _match64(D1, D2, cps, tm, rd, prior=None):
    """Matched points and SSD in 64 bits over the CPs (all inside the images)."""
    n = cps.shape[0]
    o = {"ssd": torch.empty(n, dtype=torch.float64, device=DEV), "points": torch.empty((n, 2), dtype=torch.float64, device=DEV)}
    cps, q = cps.long(), (prior.long() if prior is not None else torch.zeros_like(cps.long()))
    for N, r in sorted({(int(a), int(b)) for a, b in torch.stack([tm, rd], 1).tolist()}):
        sel = torch.nonzero((tm == N) & (rd == r)).reshape(-1)
        W, L, t0 = N + 2 * r, 2 * r + 1, N // 2
        step = max(1, int(1.5e9 / (8 * 4 * D1.shape[0] * W * W)))
        for part in sel.split(step):
            p, qq = cps[part], q[part]
            ty, tx = p[:, 1] - t0, p[:, 0] - t0
            wy, wx = ty + qq[:, 1] - r, tx + qq[:, 0] - r
            ar, aw = torch.arange(N, device=DEV), torch.arange(W, device=DEV)
            T = D1[:, (ty[:, None] + ar)[:, :, None], (tx[:, None] + ar)[:, None, :]].double()
            S = D2[:, (wy[:, None] + aw)[:, :, None], (wx[:, None] + aw)[:, None, :]].double()
            F = torch.fft.rfft2(T, s=(W, W)).conj() * torch.fft.rfft2(S)
            C = torch.fft.irfft2(F.sum(0), s=(W, W))[:, :L, :L]
            cum = torch.zeros((len(part), W + 1, W + 1), dtype=torch.float64, device=DEV)
            cum[:, 1:, 1:] = (S * S).sum(0).cumsum(1).cumsum(2)
            box = cum[:, N:, N:] - cum[:, :-N, N:] - cum[:, N:, :-N] + cum[:, :-N, :-N]
            s = (T * T).sum((0, 2, 3))[:, None, None] + box - 2 * C
            v, at = s.reshape(len(part), -1).min(1)
            vy, vx = at // L, at % L
            ox, oy = _quadratic64(s, vy, vx, r)
            o["ssd"][part] = v
            at = torch.stack([qq[:, 0] + vx - r, qq[:, 1] + vy - r], 1) + p
            o["points"][part] = at.double() + torch.stack([ox, oy], 1)
    return o


def _quadratic64(s, vy, vx, r):
    """Least-squares quadratic of the 3 x 3 scores about the minimum; none on the window's edge."""
    L = 2 * r + 1
    edge = (vy == 0) | (vy == L - 1) | (vx == 0) | (vx == L - 1)
    cy, cx = vy.clamp(1, max(1, L - 2)), vx.clamp(1, max(1, L - 2))
    b = torch.arange(len(vy), device=DEV)
    f = {(j, i): s[b, cy + j, cx + i] for j in (-1, 0, 1) for i in (-1, 0, 1)}
    s0 = sum(f.values())
    gx, gy = sum(i * v for (j, i), v in f.items()) / 6, sum(j * v for (j, i), v in f.items()) / 6
    hxy = sum(i * j * v for (j, i), v in f.items()) / 4
    hxx = 2 * (sum(i * i * v for (j, i), v in f.items()) / 2 - s0 / 3)
    hyy = 2 * (sum(j * j * v for (j, i), v in f.items()) / 2 - s0 / 3)
    det = hxx * hyy - hxy * hxy
    px, py = -(hyy * gx - hxy * gy) / det, -(hxx * gy - hxy * gx) / det
    good = (hxx > 0) & (det > 0) & (px.abs() <= 1) & (py.abs() <= 1)

    def parabola(m, c, p):
        den = m - 2 * c + p
        return torch.where(den > 0, (m - p) / (2 * den), torch.zeros_like(den)).clamp(-0.5, 0.5)
    qx, qy = parabola(f[0, -1], f[0, 0], f[0, 1]), parabola(f[-1, 0], f[0, 0], f[1, 0])
    zero = torch.zeros_like(px)
    return (torch.where(edge, zero, torch.where(good, px, qx)), torch.where(edge, zero, torch.where(good, py, qy)))


def _reject64(case, cps, res):
    ok = (res[:, 5] == 0).cpu().numpy()
    xy = cps.cpu().numpy().astype(np.float64)
    tgt = xy + res[:, 2:4].contiguous().view(torch.float32).cpu().numpy().astype(np.float64)
    lo, hi = xy[ok].min(0), xy[ok].max(0)
    c, sc = 0.5 * (lo + hi), max(0.5 * (hi - lo))
    u, v = ((xy - c) / sc).T
    mons = [np.ones_like(u), u, v, u * u, u * v, v * v, u * u * u, u * u * v, u * v * v, v * v * v]
    T = (case["degree"] + 1) * (case["degree"] + 2) // 2
    A = np.stack(mons[:T], 1)
    live = np.nonzero(ok)[0]
    while True:
        M = A[live]
        coef = np.linalg.solve(M.T @ M, M.T @ tgt[live])
        e2 = ((tgt[live] - M @ coef) ** 2).sum(1)
        rmse = math.sqrt(e2.mean())
        if rmse < case["rmse"] or len(live) - 1 < T:
            break
        live = np.delete(live, int(np.argmax(e2)))
    pad = np.zeros((2, 10))
    pad[:, :T] = coef.T
    return np.concatenate([[rmse, c[0], c[1], sc], pad[0], pad[1]])[None]


def _rectify64(case, img, cps, res, tris):
    h, w = case["h"], case["w"]
    sh, sw = img.shape
    src = img.to(torch.float64)
    pts = cps.double().cpu().numpy()
    to = pts + res[:, 2:4].contiguous().view(torch.float32).double().cpu().numpy()
    out = torch.zeros((h, w), dtype=torch.float64, device=DEV)
    done = torch.zeros((h, w), dtype=torch.bool, device=DEV)
    for t in tris.cpu().numpy():
        a, b, c = pts[t]
        x0, y0 = np.maximum(pts[t].min(0), 0).astype(int)
        x1, y1 = np.minimum(pts[t].max(0), [w - 1, h - 1]).astype(int)
        if x0 > x1 or y0 > y1:
            continue
        X = torch.arange(x0, x1 + 1, device=DEV, dtype=torch.float64)[None, :]
        Y = torch.arange(y0, y1 + 1, device=DEV, dtype=torch.float64)[:, None]

        def side(p, q):
            return (q[0] - p[0]) * (Y - p[1]) - (q[1] - p[1]) * (X - p[0])
        wa, wb, wc = side(b, c), side(c, a), side(a, b)
        area = (b[0] - a[0]) * (c[1] - a[1]) - (b[1] - a[1]) * (c[0] - a[0])
        box = (slice(int(y0), int(y1) + 1), slice(int(x0), int(x1) + 1))
        inside = (wa >= 0) & (wb >= 0) & (wc >= 0) & ~done[box]
        U = (wa * to[t[0], 0] + wb * to[t[1], 0] + wc * to[t[2], 0]) / area
        V = (wa * to[t[0], 1] + wb * to[t[1], 1] + wc * to[t[2], 1]) / area
        iu, iv = U.floor().clamp(0, sw - 1).long(), V.floor().clamp(0, sh - 1).long()
        iu1, iv1 = (iu + 1).clamp(max=sw - 1), (iv + 1).clamp(max=sh - 1)
        fu, fv = U - iu, V - iv
        val = (src[iv, iu] * (1 - fu) + src[iv, iu1] * fu) * (1 - fv) + (src[iv1, iu] * (1 - fu) + src[iv1, iu1] * fu) * fv
        hit = inside & (U >= 0) & (U <= sw - 1) & (V >= 0) & (V <= sh - 1)
        out[box] = torch.where(hit, val, out[box])
        done[box] |= inside
    return out


def exact(case, seed):
    k = case["kind"]
    if k == "detect":         # pixel positions only: whole numbers
        return None
    if k == "extract":
        D = _cfog64(_image(seed, case["h"], case["w"], case["dtype"]), case["m"], case["radius"], case["orient"])
        return {"volume": D, "sqnorm": (D * D).sum(0)}
    none = {"dx": None, "dy": None, "status": None}
    if k in ("pair", "step", "fhog"):
        s = case["size"]
        A, B, _, _ = _pair(seed, s, s, "shift" if k == "pair" else "speckle")
        D1, D2 = (_fhog64(i, case["cell"]) if k == "fhog" else _cfog64(i) for i in (A, B))
        cps = _grid_cps(case) if k == "pair" else _harris64(A, case["grid"], _margin(case))
        tm, rd = _class_rows(case, seed, case["grid"] ** 2)
        out = {"match": {**none, **_match64(D1, D2, cps, tm, rd)}}
        if k == "pair" or k == "fhog":
            out["ref"], out["sen"] = D1, D2
        if k != "pair":
            out["cps"] = None
        return out
    if k == "match":
        pairs, cps, job, prior = _match_images(case, seed)
        tm, rd = _class_rows(case, seed, cps.shape[0])
        n = cps.shape[0]
        out = {"ssd": torch.empty(n, dtype=torch.float64, device=DEV), "points": torch.empty((n, 2), dtype=torch.float64, device=DEV)}
        for j, (A, B, _, _) in enumerate(pairs):
            at = torch.nonzero(job == j).reshape(-1) if job is not None else torch.arange(n, device=DEV)
            o = _match64(_cfog64(A), _cfog64(B), cps[at], tm[at], rd[at], prior[at] if prior is not None else None)
            for q in out:
                out[q][at] = o[q]
        return {"match": {**none, **out}}
    if k == "reject":
        cps, res = _reject_inputs(case, seed)
        return {"keep": None, "order": None, "counts": None, "model": _reject64(case, cps, res)}
    img, cps, res = _rectify_inputs(case, seed)
    # the triangulation is an input of the call, like the CPs
    return {"image": _rectify64(case, img, cps, res, torch.from_numpy(P.tin_delaunay(cps)))}
