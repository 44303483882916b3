"""Workloads the library is measured on: what they are, their inputs, one pass, and what a pass cannot do without.

The sizes are those of the synthetic workloads in ``synth/scenes.py`` (160x120 grey, 640x480, 1280x960 and
1920x1080 RGB, the uneven batch of 320x240..1024x768 pairs), plus odd and ragged sizes in between.  Inputs are layered textured scenes rendered on the GPU by ``_scene`` with
the same recipe as ``synth/scenes.py`` (slanted planes with rectangular or elliptical footprints, value-noise
textures, sensor noise), so that a case can be prepared many times.

A case's "kind" is the entry point:
  disparity   Context.compute_disparity: both maps of one pair, in the context's precision
  cost        Context.cost_volume: the FP32 matching-cost volume
  aggregate   Context.aggregate: aggregated volume and both maps of a cost volume the caller made
  batch       fbs_compute_disparity_batched: many uneven pairs in one call
  lr          fbs_compute_disparity_lr: both views and the consistency check
  learned     fbs_compute_disparity_learned: network proposal, then the band-restricted path
  net         fbs_band_net_forward: the network's outputs, centre and confidence of one pair
"""

import math
import os
import random

import numpy as np
import torch
import torch.nn.functional as F

import paper_1807_02044_gb300 as fbs

_ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
_PREC = {"f32": fbs.FBS_PREC_F32, "bf16": fbs.FBS_PREC_BF16, "f16": fbs.FBS_PREC_F16}
_COST = {"ncc": fbs.FBS_COST_NCC, "tad": fbs.FBS_COST_TAD}
_HALF_BAND = 8          # band half-width of the shipped network


def _case(kind, H, W, D, radius, C=3, prec="f32", cost="ncc", sigma_s=None, sigma_r=12.0, tau=30.0, **more):
    return dict(kind=kind, H=H, W=W, C=C, D=D, radius=radius, prec=prec, cost=cost,
                sigma_s=float(radius if sigma_s is None else sigma_s), sigma_r=sigma_r, tau=tau, **more)


def listed():
    return [
        # a small grey camera pair in FP32 (the smallest call: launches and latency count)
        dict(_case("disparity", 120, 160, 16, 4, C=1, sigma_r=10.0, tau=20.0), name="gray160x120_f32"),
        # the benchmark pair: one VGA colour frame, FP32 and with 16-bit operands on the tensor cores
        dict(_case("disparity", 480, 640, 64, 7), name="vga_f32"),
        dict(_case("disparity", 480, 640, 64, 7, prec="bf16"), name="vga_bf16"),
        # a larger frame with a wide window, FP16 operands
        dict(_case("disparity", 960, 1280, 128, 15, prec="f16"), name="960p_f16"),
        # full HD over 256 disparities, BF16 operands
        dict(_case("disparity", 1080, 1920, 256, 9, prec="bf16"), name="hd_bf16"),
        # a ragged frame with the truncated absolute difference, D no multiple of a vector or tile
        dict(_case("disparity", 575, 767, 93, 11, cost="tad"), name="ragged_tad_f32"),
        # the matching cost alone (a caller that aggregates in its own way), odd width
        dict(_case("cost", 479, 641, 70, 0, sigma_s=1.0), name="cost_641x479"),
        # aggregation of the caller's own cost volume, the aggregated volume returned
        dict(_case("aggregate", 375, 450, 60, 9), name="aggregate_450x375"),
        # a server's batch: pairs of uneven size, disparity range and radius in one call
        dict(_case("batch", 768, 1024, 192, 11, prec="bf16", pairs=24, mix=0), name="batch24_bf16"),
        # both views and the left-right check of a VGA pair
        dict(_case("lr", 480, 640, 64, 7), name="lr_vga_f32"),
        # the learned band proposal on full HD (network, bands, band-restricted FP32 path)
        dict(_case("learned", 1080, 1920, 256, 9), name="learned_hd"),
        # the proposal network alone on a crop of the size it is trained on
        dict(_case("net", 640, 1280, 256, 9), name="net_1280x640"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes log-uniform over the listed range (odd ones among them), any D and radius of the range;
    frames are shrunk until the pass costs no more than the largest listed case of its arithmetic."""
    kind = rng.choice(["disparity"] * 6 + ["cost", "aggregate", "batch", "lr", "learned", "net"])
    prec = "f32" if kind in ("cost", "learned", "net") else rng.choice(["f32", "f32", "bf16", "f16"])
    H, W = _log(rng, 60, 1080), _log(rng, 80, 1920)
    D, radius = _log(rng, 8, 256), rng.randint(1, 15)
    C = rng.choice([1, 3, 3])
    cost = "ncc" if kind in ("learned", "net", "aggregate") else rng.choice(["ncc", "ncc", "ncc", "tad"])
    more = {}
    if kind == "batch":
        H, W, D, radius, more = 768, 1024, 192, 11, dict(pairs=rng.randint(2, 20), mix=rng.randint(1, 10 ** 6))
    if kind in ("learned", "net"):
        H, W, D, radius = max(H, 120), max(W, 160), max(32, D), min(radius, 9)
    if kind == "cost":
        radius = 0
    c = _case(kind, H, W, D, radius, C=C, prec=prec, cost=cost, sigma_s=max(1.0, float(radius)),
              sigma_r=float(rng.choice([8, 10, 12, 16, 24])), tau=float(rng.choice([20, 30])), **more)
    if kind in ("disparity", "lr", "aggregate", "cost"):
        most_taps, most_costs = (5e10 if prec == "f32" else 1.8e11), (5.3e8 if kind in ("disparity", "lr") else 2.5e8)
        while _taps(c) * (2 if kind == "lr" else 1) > most_taps or c["H"] * c["W"] * c["D"] > most_costs:
            c["H"], c["W"] = int(c["H"] * 0.85), int(c["W"] * 0.85)
    return c


def _taps(c):
    return float(c["H"]) * c["W"] * c["D"] * (2 * c["radius"] + 1) ** 2


def _members(case):
    """Shapes of a batch: W and H uniform in 320..1024 x 240..768, D and radius from the batch workload's sets."""
    rng = random.Random(case["mix"])
    return [dict(case, kind="disparity", H=rng.randint(240, case["H"]), W=rng.randint(320, case["W"]),
                 D=rng.choice([32, 64, 128, 192]), radius=(r := rng.choice([4, 7, 11])), sigma_s=float(r))
            for _ in range(case["pairs"])]


# ---- inputs ----------------------------------------------------------------------------------------------------
def _texture(g, C, H, W, uniform):
    """A texture of H x W pixels, C channels, in [0, 255]: uniform noise, or five octaves of bilinear value noise
    (finest cell 2 px) stretched to the full range."""
    if uniform:
        return torch.rand((1, C, H, W), generator=g, device="cuda") * 255.0
    out, total = 0.0, 0.0
    for o in range(5):
        cell = 2 ** (5 - o)
        grid = torch.rand((1, C, H // cell + 3, W // cell + 3), generator=g, device="cuda")
        up = F.interpolate(grid, scale_factor=cell, mode="bilinear", align_corners=False)
        out = out + 0.55 ** o * up[:, :, cell // 2:cell // 2 + H, cell // 2:cell // 2 + W]
        total += 0.55 ** o
    return torch.clamp(0.5 + (out / total - 0.5) * 2.6, 0.0, 1.0) * 255.0


def _scene(case, seed):
    """A stereo pair of layered slanted planes: (left, right), uint8 HWC on the GPU."""
    H, W, C, D = case["H"], case["W"], case["C"], case["D"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = random.Random(seed)
    hi = float(D - 1)
    y, x = torch.meshgrid(torch.arange(H, device="cuda", dtype=torch.float32),
                          torch.arange(W, device="cuda", dtype=torch.float32), indexing="ij")
    TH, TW = H + 8, W + D + 16
    views = [dict(img=torch.zeros((C, H, W), device="cuda"), d=torch.full((H, W), -1e9, device="cuda")) for _ in range(2)]
    for k in range(r.randint(3, 6)):
        lo_k, hi_k = (0.0, 0.35 * hi) if k == 0 else (r.uniform(0.2, 0.6) * hi, 0.0)
        if k:
            hi_k = min(hi, lo_k + r.uniform(0.1, 0.4) * hi)
        d00, d10 = r.uniform(lo_k, hi_k), r.uniform(lo_k, hi_k)
        d01 = min(max(r.uniform(lo_k, hi_k), lo_k + d00 - d10), hi_k + d00 - d10)
        a, b, c = max(-0.5, min(0.5, (d10 - d00) / W)), (d01 - d00) / H, d00
        cx, cy = r.uniform(0.15, 0.85) * W, r.uniform(0.15, 0.85) * H
        rx, ry, ellipse = r.uniform(0.1, 0.28) * W, r.uniform(0.1, 0.28) * H, r.random() < 0.5
        tex = _texture(g, C, TH, TW, C == 1)
        for view, v in enumerate(views):
            xl = x if view == 0 else (x + b * y + c) / (1.0 - a)    # left coordinate of the surface point seen here
            d = a * xl + b * y + c
            u, w = (xl - cx) / rx, (y - cy) / ry
            inside = torch.ones_like(x, dtype=torch.bool) if k == 0 else \
                (u * u + w * w <= 1.0 if ellipse else (u.abs() <= 1.0) & (w.abs() <= 1.0))
            m = inside & (d > v["d"])
            grid = torch.stack([(xl + 2.5) * (2.0 / TW) - 1.0, (y + 2.5) * (2.0 / TH) - 1.0], -1)[None]
            val = F.grid_sample(tex, grid, mode="bilinear", padding_mode="border", align_corners=False)[0]
            v["img"], v["d"] = torch.where(m, val, v["img"]), torch.where(m, d, v["d"])
    out = []
    for v in views:
        noisy = v["img"] + 2.0 * torch.randn(v["img"].shape, generator=g, device="cuda")
        out.append(noisy.round().clamp(0, 255).to(torch.uint8).permute(1, 2, 0).contiguous())
    return out[0], out[1]


def _own_cost(left, right, D):
    """A caller's own cost volume: mean absolute colour difference, truncated at 40 and scaled to [0, 1]."""
    H, W, _ = left.shape
    L, R = left.float(), right.float()
    out = torch.full((H, W, D), 1.0, device="cuda")
    for d in range(min(D, W)):
        out[:, d:, d] = (L[:, d:] - R[:, :W - d]).abs().mean(-1).clamp(max=40.0) / 40.0
    return out


def prepare(case, seed):
    ctx = fbs.Context(0, cost=_COST[case["cost"]], prec=_PREC[case["prec"]])
    s = dict(case=case, ctx=ctx)
    kind = case["kind"]
    if kind == "batch":
        pairs = []
        for i, m in enumerate(_members(case)):
            left, right = _scene(m, seed * 1009 + i)
            pairs.append(dict(left=left, right=right, disp_int=_map(m, torch.int32), disp_subpix=_map(m, torch.float32),
                              **_params(m)))
        s.update(pairs=pairs, table=fbs.make_pairs(pairs))
        return s
    left, right = _scene(case, seed)
    s.update(left=left, right=right)
    if kind == "aggregate":
        s["cost"] = _own_cost(left, right, case["D"])
    if kind == "lr":
        s["maps"] = [_map(case, t) for t in (torch.int32, torch.float32) * 2]
    if kind in ("learned", "net"):
        fbs.fbs_band_net_load(ctx.ctx, fbs.default_band_net_path())
    if kind == "learned":
        s["theta"] = fbs.default_band_threshold()
        s["pair"] = dict(left=left, right=right, disp_int=_map(case, torch.int32), disp_subpix=_map(case, torch.float32),
                         **_params(case))
    if kind == "net":
        s["out_q"] = torch.empty(((case["H"] + 3) // 4, (case["W"] + 3) // 4, 2), device="cuda")
        s["planes"] = [_map(case, torch.float32) for _ in range(2)]
    return s


def _map(c, dtype):
    return torch.empty((c["H"], c["W"]), dtype=dtype, device="cuda")


def _params(c):
    return {k: c[k] for k in ("H", "W", "C", "D", "radius", "sigma_s", "sigma_r", "tau")}


def run(s):
    c, ctx = s["case"], s["ctx"]
    kind = c["kind"]
    st = torch.cuda.current_stream()
    if kind == "disparity":
        return ctx.compute_disparity(s["left"], s["right"], c["D"], c["radius"], c["sigma_s"], c["sigma_r"], c["tau"])
    if kind == "cost":
        return ctx.cost_volume(s["left"], s["right"], c["D"], c["tau"])
    if kind == "aggregate":
        return ctx.aggregate(s["cost"], s["left"], c["radius"], c["sigma_s"], c["sigma_r"])
    if kind == "batch":
        fbs.fbs_compute_disparity_batched(ctx.ctx, s["table"], st)
        return [(p["disp_int"], p["disp_subpix"]) for p in s["pairs"]]
    if kind == "lr":
        fbs.fbs_compute_disparity_lr(ctx.ctx, s["left"], s["right"], c["H"], c["W"], c["C"], c["D"], c["radius"],
                                     c["sigma_s"], c["sigma_r"], c["tau"], *s["maps"], True, st)
        return s["maps"]
    if kind == "learned":
        fbs.fbs_compute_disparity_learned(ctx.ctx, s["pair"], _HALF_BAND, s["theta"], st)
        return [s["pair"]["disp_int"], s["pair"]["disp_subpix"]]
    fbs.fbs_band_net_forward(ctx.ctx, s["left"], s["right"], c["H"], c["W"], c["C"], c["D"], s["out_q"], *s["planes"], st)
    return [s["out_q"], *s["planes"]]


def work(case):
    """Bytes: images (or the caller's volume) in, maps (or volumes) out, once each.  Flops: one multiply-add per pixel,
    disparity and window tap, and nine per matching cost; for the learned form only the bands of +-8 disparities."""
    kind = case["kind"]
    if kind == "batch":
        parts = [work(m) for m in _members(case)]
        return {k: float(sum(p[k] for p in parts)) for k in ("bytes", "flops")}
    px = float(case["H"]) * case["W"]
    images, maps, volume, taps = 2 * px * case["C"], 8 * px, 4 * px * case["D"], _taps(case)
    costs = px * case["D"]
    if kind == "cost":
        return dict(bytes=images + volume, flops=18 * costs)
    if kind == "aggregate":
        return dict(bytes=volume * 2 + px * case["C"] + maps, flops=2 * taps)
    if kind == "lr":
        return dict(bytes=images + 2 * maps, flops=4 * taps + 18 * costs)
    net = px / 16 * 2 * 9 * (6 * 32 + 4 * 32 * 32 + 32 * 2)
    if kind == "learned":
        share = min(1.0, (2 * _HALF_BAND + 1) / case["D"])
        return dict(bytes=images + maps, flops=(2 * taps + 18 * costs) * share + net)
    if kind == "net":
        return dict(bytes=images + maps + px / 2, flops=net + px / 16 * case["D"] / 4 * 18)
    return dict(bytes=images + maps, flops=2 * taps + 18 * costs)


# ---- the same in 64 bits, from the definitions -------------------------------------------------------------------
def _grey(img):
    return img.double().sum(-1)


def _box(p, H, W):
    """3x3 sums of a plane padded by one pixel on each side."""
    return sum(p[j:j + H, i:i + W] for j in range(3) for i in range(3))


def _ncc_volume(gl, gr, D):
    """1 - normalised correlation of the clamped 3x3 blocks of two planes; 1 for a flat block, 2 where x < d."""
    H, W = gl.shape
    pl, pr = (F.pad(g[None, None], (1, 1, 1, 1), mode="replicate")[0, 0] for g in (gl, gr))
    Sl, Sr = _box(pl, H, W), _box(pr, H, W)
    Vl, Vr = 9 * _box(pl * pl, H, W) - Sl * Sl, 9 * _box(pr * pr, H, W) - Sr * Sr
    out = torch.full((H, W, D), 2.0, dtype=torch.float64, device="cuda")
    for d in range(min(D, W)):
        n = W - d
        num = 9 * _box(pl[:, d:] * pr[:, :n + 2], H, n) - Sl[:, d:] * Sr[:, :n]
        v = Vl[:, d:] * Vr[:, :n]
        out[:, d:, d] = 1.0 - torch.where(v > 0, num / v.clamp(min=1e-300).sqrt(), torch.zeros_like(num))
    return out


def _cost64(left, right, c):
    if c["cost"] == "ncc":
        return _ncc_volume(_grey(left), _grey(right), c["D"])
    H, W, _ = left.shape
    L, R = left.double(), right.double()
    out = torch.full((H, W, c["D"]), c["tau"], dtype=torch.float64, device="cuda")
    for d in range(min(c["D"], W)):
        out[:, d:, d] = (L[:, d:] - R[:, :W - d]).abs().mean(-1).clamp(max=c["tau"])
    return out


def _aggregate64(cost, guide, c):
    H, W, _ = cost.shape
    G = guide.double()
    acc, den = torch.zeros_like(cost), torch.zeros((H, W), dtype=torch.float64, device="cuda")
    r = c["radius"]
    for dy in range(-min(r, H - 1), min(r, H - 1) + 1):
        for dx in range(-min(r, W - 1), min(r, W - 1) + 1):
            p = (slice(max(0, -dy), H - max(0, dy)), slice(max(0, -dx), W - max(0, dx)))
            q = (slice(max(0, dy), H + min(0, dy)), slice(max(0, dx), W + min(0, dx)))
            w = torch.exp(-(dx * dx + dy * dy) / c["sigma_s"] ** 2
                          - (G[q] - G[p]).square().sum(-1) / c["sigma_r"] ** 2)
            den[p] += w
            acc[p].addcmul_(w[..., None], cost[q])
    return acc.div_(den[..., None])


def _subpixel64(A, lo=None, hi=None):
    """Winner (smallest d) and parabola vertex per pixel, over each pixel's [lo, hi] (default: all)."""
    D = A.shape[2]
    if lo is not None:
        ds = torch.arange(D, device="cuda")
        A = torch.where((ds >= lo[..., None]) & (ds <= hi[..., None]), A, torch.full_like(A, math.inf))
    best = A.argmin(2)
    take = lambda k: A.gather(2, (best + k).clamp(0, D - 1)[..., None])[..., 0]  # noqa: E731
    m, z, p = take(-1), take(0), take(1)
    den = 2 * m + 2 * p - 4 * z
    lo, hi = (0, D - 1) if lo is None else (lo, hi)
    ok = (best > lo) & (best < hi) & (den > 0)
    return best, best + torch.where(ok, (m - p) / torch.where(ok, den, torch.ones_like(den)), torch.zeros_like(den))


def _view64(left, right, c):
    return _subpixel64(_aggregate64(_cost64(left, right, c), left, c))


def _net_params():
    path = os.path.join(_ROOT, "paper_1807_02044_gb300", "band_net_1920x1080_d256.bin")
    return torch.from_numpy(np.fromfile(path, np.float32, offset=12)).double().cuda()


def _net64(theta, left, right, c):
    """Quarter-resolution features and the six 3x3 convolutions: (e*, outputs [2][Hq][Wq])."""
    H, W, C, Dq = c["H"], c["W"], c["C"], (c["D"] + 3) // 4
    Hq, Wq = (H + 3) // 4, (W + 3) // 4
    quarter = [F.pad(_grey(i)[None, None], (0, 4 * Wq - W, 0, 4 * Hq - H), mode="replicate")[0, 0]
               .reshape(Hq, 4, Wq, 4).sum((1, 3)) for i in (left, right)]
    K = _ncc_volume(*quarter, Dq).permute(2, 0, 1)[:, None]
    ones = torch.ones((1, 1, 5, 5), dtype=torch.float64, device="cuda")
    K = (F.conv2d(K, ones, padding=2) / F.conv2d(torch.ones_like(K[:1]), ones, padding=2))[:, 0].permute(1, 2, 0)
    e = K.argmin(2)
    at = lambda k: torch.where((e + k >= 0) & (e + k < Dq), K.gather(2, (e + k).clamp(0, Dq - 1)[..., None])[..., 0],  # noqa: E731
                               torch.full_like(K[..., 0], 2.0))
    far = (torch.arange(Dq, device="cuda") - e[..., None]).abs() >= 2
    k1, k2 = at(0), torch.where(far, K, torch.full_like(K, 2.0)).amin(2).clamp(max=2.0)
    X = torch.stack([quarter[0] / (16 * 255 * C) - 0.5, e / Dq, k1, (k2 - k1).clamp(max=1.0), at(-1) - k1, at(1) - k1])[None]
    o = 0
    for layer in range(6):
        ci, co = (6 if layer == 0 else 32), (2 if layer == 5 else 32)
        w = theta[o:o + 9 * ci * co].reshape(3, 3, ci, co).permute(3, 2, 0, 1)
        o += 9 * ci * co
        X = F.conv2d(X, w, theta[o:o + co], padding=1)
        o += co
        X = X if layer == 5 else F.relu(X)
    return e, X[0]


def _proposal64(left, right, c):
    """The network's outputs [Hq][Wq][2] and the full-resolution centre and confidence."""
    e, out = _net64(_net_params(), left, right, c)
    up = lambda q: q.repeat_interleave(4, 0).repeat_interleave(4, 1)[:c["H"], :c["W"]]  # noqa: E731
    return out.permute(1, 2, 0), up(4 * (e + out[0])), up(torch.sigmoid(out[1]))


def _learned64(left, right, c, threshold):
    _, centre, conf = _proposal64(left, right, c)
    m = torch.floor(centre + 0.5).clamp(0, c["D"] - 1).long()
    sure = conf >= threshold
    lo = torch.where(sure, (m - _HALF_BAND).clamp(min=0), torch.zeros_like(m))
    hi = torch.where(sure, (m + _HALF_BAND).clamp(max=c["D"] - 1), torch.full_like(m, c["D"] - 1))
    return _subpixel64(_aggregate64(_cost64(left, right, c), left, c), lo, hi)[1]


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return [(None, _view64(*_scene(m, seed * 1009 + i), m)[1]) for i, m in enumerate(_members(case))]
    left, right = _scene(case, seed)
    if kind == "disparity":
        return None, _view64(left, right, case)[1]
    if kind == "cost":
        return _cost64(left, right, case)
    if kind == "aggregate":
        A = _aggregate64(_own_cost(left, right, case["D"]).double(), left, case)
        return A, None, _subpixel64(A)[1]
    if kind == "lr":
        dl, sl = _view64(left, right, case)
        dr, sr = (v.flip(1) for v in _view64(right.flip(1).contiguous(), left.flip(1).contiguous(), case))
        u = torch.arange(case["W"], device="cuda") - dl
        keep = (u >= 0) & (dr.gather(1, u.clamp(min=0)) == dl)
        return [None, torch.where(keep, sl, torch.full_like(sl, -1.0)), None, sr]
    if kind == "learned":
        return [None, _learned64(left, right, case, fbs.default_band_threshold())]
    return list(_proposal64(left, right, case))
