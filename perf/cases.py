"""Workloads of the TV library, each one call (or one call sequence) that a user's program makes.

Every case goes through the public Python entry points on inputs that are resident on the GPU.
Inputs are drawn on the device from a seed: noisy step signals, noisy images of rectangles and
disks, impulse-noise images and matching-cost volumes, with the distributions of
``paper_1502_07770_gb300.synth``. ``exact`` restates each problem in float64 with plain torch.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1502_07770_gb300 import (chain_prox, chain_prox_backward, chain_prox_nonconvex, learned,
                                    synth, tv2d_denoise, tv2d_denoise_batched, tv2d_denoise_l1)

DEV = "cuda:0"
TOL = 1e-4        # per-pixel primal-dual gap of the ROF cases
MAX_ITERS = 200


def listed():
    return [
        # the rows and columns of one 256 x 256 image: the smallest batch, launch and latency count
        {"name": "chains_512x256", "kind": "chains", "chains": 512, "nodes": 256, "lam": 0.2,
         "edges": False},
        # throughput: many signals of one length with one weight
        {"name": "chains_65536x1024", "kind": "chains", "chains": 65536, "nodes": 1024,
         "lam": 0.15, "edges": False},
        # signals of uneven length (CSR offsets) with a weight per edge
        {"name": "chains_ragged_edges", "kind": "ragged", "chains": 6000, "longest": 2500,
         "size_seed": 5, "lam": 0.2},
        # the forward pass of a prox layer on a training batch, learnable weight per edge,
        # a length that is no multiple of anything
        {"name": "layer_forward_edges", "kind": "chains", "chains": 4096, "nodes": 1023,
         "lam": 0.15, "edges": True},
        # the backward pass of a prox layer: gradients of the input and of the edge weights
        {"name": "layer_backward_4096x1024", "kind": "backward", "chains": 4096, "nodes": 1024,
         "edges": True},
        # one photograph-sized image to a gap of 1e-4, from zero
        {"name": "rof_1024", "kind": "rof", "height": 1024, "width": 1024, "shapes": 200,
         "lam": 0.1, "edges": False},
        # a small image of odd size with edge-aware weights: latency
        {"name": "rof_edges_297x401", "kind": "rof", "height": 297, "width": 401, "shapes": 60,
         "lam": 0.2, "edges": True},
        # a batch of images of uneven sizes with edge-aware weights, as a service denoises them
        {"name": "rof_batch_64", "kind": "batch", "images": 64, "size_seed": 100, "edges": True},
        # one image from the network's dual: inference and the solve
        {"name": "rof_warm_1024", "kind": "warm", "height": 1024, "width": 1024, "shapes": 200,
         "lam": 0.1},
        # a training step's forward and backward of the warm-start network
        {"name": "net_train_8x512", "kind": "train", "images": 8, "height": 512, "width": 512},
        # impulse noise: TV-l1, a fixed number of iterations
        {"name": "l1_768x1024", "kind": "l1", "height": 768, "width": 1024, "iters": 60,
         "lam": 0.55},
        # scanlines of a stereo pair: truncated TV on a cost volume
        {"name": "stereo_1000x1482x126", "kind": "stereo", "rows": 1000, "nodes": 1482,
         "labels": 126},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["chains", "chains", "ragged", "backward", "rof", "rof", "batch", "warm",
                       "train", "l1", "stereo"])
    if kind == "chains":
        n = _log(rng, 128, 4096)
        if rng.random() < 0.5:
            n = (n + 3) // 4 * 4
        return {"kind": kind, "chains": _log(rng, 256, min(65536, (1 << 26) // n)), "nodes": n,
                "lam": round(rng.uniform(0.05, 0.3), 3), "edges": rng.random() < 0.5}
    if kind == "ragged":
        return {"kind": kind, "chains": _log(rng, 300, 12000), "longest": _log(rng, 200, 4000),
                "size_seed": rng.randrange(1 << 20), "lam": round(rng.uniform(0.05, 0.3), 3)}
    if kind == "backward":
        return {"kind": kind, "chains": _log(rng, 512, 16384), "nodes": _log(rng, 256, 2048),
                "edges": rng.random() < 0.5}
    if kind == "rof":
        return {"kind": kind, "height": _log(rng, 200, 1600), "width": _log(rng, 200, 1600),
                "shapes": rng.randrange(40, 201), "lam": round(rng.uniform(0.05, 0.3), 3),
                "edges": rng.random() < 0.5}
    if kind == "batch":
        return {"kind": kind, "images": rng.randrange(4, 49),
                "size_seed": rng.randrange(1 << 20), "edges": rng.random() < 0.5}
    if kind == "warm":
        return {"kind": kind, "height": _log(rng, 256, 1100), "width": _log(rng, 256, 1100),
                "shapes": 200, "lam": round(rng.uniform(0.05, 0.3), 3)}
    if kind == "train":
        return {"kind": kind, "images": rng.randrange(2, 9), "height": rng.randrange(128, 513),
                "width": rng.randrange(128, 513)}
    if kind == "l1":
        return {"kind": kind, "height": _log(rng, 200, 1024), "width": _log(rng, 200, 1024),
                "iters": rng.randrange(20, 61), "lam": round(rng.uniform(0.4, 0.7), 3)}
    return {"kind": "stereo", "rows": _log(rng, 100, 1000), "nodes": rng.randrange(300, 1483),
            "labels": rng.randrange(32, 127)}


# ------------------------------------------------------------------ inputs --
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) & 0x7FFFFFFFFFFF)


def _signals(rows, n, gen, seg_lo=8, seg_hi=64, noise=0.1):
    """(rows, n) noisy step signals: segments of U{8..64} nodes, levels U[0, 1]."""
    segs = n // seg_lo + 1
    ends = torch.randint(seg_lo, seg_hi + 1, (rows, segs), generator=gen, device=DEV,
                         dtype=torch.int32).cumsum(1)
    mark = torch.zeros((rows, n + 1), dtype=torch.int32, device=DEV)
    mark.scatter_(1, ends.clamp_(max=n).long(), 1)
    seg = mark[:, :n].cumsum(1)
    level = torch.rand((rows, segs + 1), generator=gen, device=DEV)
    y = level.gather(1, seg)
    return y.add_(torch.randn((rows, n), generator=gen, device=DEV), alpha=noise)


def _lengths(case):
    rng = np.random.Generator(np.random.PCG64(case["size_seed"]))
    return rng.integers(1, case["longest"] + 1, size=case["chains"])


def _image(H, W, shapes, seed, noise=0.1):
    """A noisy image of random rectangles and disks (levels U[0, 1]) on a grey ground."""
    rng = random.Random(seed)
    img = torch.full((H, W), 0.5, device=DEV)
    rr = torch.arange(H, device=DEV, dtype=torch.float32)[:, None]
    cc = torch.arange(W, device=DEV, dtype=torch.float32)[None, :]
    for _ in range(shapes):
        level, cy, cx = rng.random(), rng.uniform(0, H), rng.uniform(0, W)
        if rng.random() < 0.5:
            hh, hw = 0.5 * rng.uniform(H / 32, H / 4), 0.5 * rng.uniform(W / 32, W / 4)
            img[max(0, int(cy - hh)):int(cy + hh) + 1, max(0, int(cx - hw)):int(cx + hw) + 1] = level
        else:
            rad = rng.uniform(W / 64, W / 8)
            ys = slice(max(0, int(cy - rad)), min(H, int(cy + rad) + 2))
            xs = slice(max(0, int(cx - rad)), min(W, int(cx + rad) + 2))
            inside = (rr[ys] - cy).square() + (cc[:, xs] - cx).square() <= rad * rad
            img[ys, xs].masked_fill_(inside, level)
    return img.add_(torch.randn((H, W), generator=_gen(seed), device=DEV), alpha=noise)


def _edge_weights(f, lam, scale=0.2):
    wh = lam * torch.exp(-(f[:, 1:] - f[:, :-1]).abs() / scale)
    wv = lam * torch.exp(-(f[1:] - f[:-1]).abs() / scale)
    return wh.contiguous(), wv.contiguous()


def _batch_inputs(case, seed):
    sizes, lams = synth.uneven_image_sizes(case["images"], case["size_seed"])
    fs = [_image(h, w, 200, seed * 1009 + m) for m, (h, w) in enumerate(sizes)]
    if not case["edges"]:
        return fs, lams, None, None
    ws = [_edge_weights(f, lam) for f, lam in zip(fs, lams)]
    return fs, lams, [w[0] for w in ws], [w[1] for w in ws]


def _rof_inputs(case, seed):
    f = _image(case["height"], case["width"], case["shapes"], seed)
    wh, wv = _edge_weights(f, case["lam"]) if case.get("edges") else (None, None)
    return f, wh, wv


def _train_inputs(case, seed):
    B, H, W = case["images"], case["height"], case["width"]
    rng = random.Random(seed)
    lam = torch.tensor([rng.uniform(0.05, 0.3) for _ in range(B)], device=DEV)
    f = torch.stack([_image(H, W, 200, seed * 31 + m) for m in range(B)])
    # targets: duals D_v^T p of smooth fields |p| <= lambda
    coarse = torch.randn((B, 1, (H + 15) // 16, (W + 15) // 16), generator=_gen(seed), device=DEV)
    p = torch.nn.functional.interpolate(coarse, size=(H, W), mode="nearest")[:, 0]
    p = lam[:, None, None] * torch.tanh(p)
    p[:, -1] = 0
    target = -p
    target[:, 1:] += p[:, :-1]
    return f, lam, target.contiguous()


def _volume(case, seed):
    """Truncated-linear matching costs around a piecewise-constant disparity, with noise and
    false minima at 10 % of the pixels."""
    R, n, L = case["rows"], case["nodes"], case["labels"]
    gen = _gen(seed)
    d = _signals(R, n, gen, 16, 200, 0.0).mul_(L - 1)
    lab = torch.arange(L, device=DEV, dtype=torch.float32)
    cost = (lab - d[..., None]).abs_().mul_(0.25).clamp_(max=1.0)
    cost.add_(torch.rand((R, n, L), generator=gen, device=DEV), alpha=0.3)
    false = torch.randint(0, L, (R, n), generator=gen, device=DEV).float()
    hit = (torch.rand((R, n), generator=gen, device=DEV) < 0.1).float()
    dip = (lab - false[..., None]).abs_().mul_(-0.25).add_(0.5).clamp_(min=0.0)
    return cost.sub_(dip.mul_(hit[..., None]))


STEREO_W, STEREO_C = 0.125, 1.0   # C / w = 8 exactly


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "chains":
        gen = _gen(seed)
        s["y"] = _signals(case["chains"], case["nodes"], gen)
        if case["edges"]:
            s["w"] = case["lam"] * (0.2 + 0.8 * torch.rand(s["y"].shape, generator=gen, device=DEV))
        s["x"] = torch.empty_like(s["y"])
    elif kind == "ragged":
        gen = _gen(seed)
        lengths = _lengths(case)
        offsets = np.zeros(len(lengths) + 1, dtype=np.int64)
        offsets[1:] = np.cumsum(lengths)
        total = int(offsets[-1])
        s["y"] = _signals(-(-total // 4096), 4096, gen).reshape(-1)[:total].contiguous()
        s["w"] = case["lam"] * (0.2 + 0.8 * torch.rand(total, generator=gen, device=DEV))
        s["offsets"] = torch.from_numpy(offsets).to(DEV)
        s["max_len"] = int(lengths.max())
        s["x"] = torch.empty_like(s["y"])
    elif kind == "backward":
        gen = _gen(seed)
        shape = (case["chains"], case["nodes"])
        # a solution: runs of equal values, single nodes up to long plateaus
        s["x"] = _signals(*shape, gen, 2, 40, 0.0)
        s["grad"] = torch.randn(shape, generator=gen, device=DEV)
    elif kind == "rof":
        s["f"], s["wh"], s["wv"] = _rof_inputs(case, seed)
    elif kind == "batch":
        s["fs"], s["lams"], s["whs"], s["wvs"] = _batch_inputs(case, seed)
    elif kind == "warm":
        s["f"] = _rof_inputs(case, seed)[0]
        s["net"] = learned.load_weights(DEV)
        s["lam_t"] = torch.tensor([case["lam"]], dtype=torch.float32, device=DEV)
    elif kind == "train":
        s["net"] = learned.load_weights(DEV)
        s["f"], s["lam"], s["target"] = _train_inputs(case, seed)
    elif kind == "l1":
        f = _image(case["height"], case["width"], 200, seed)
        gen = _gen(seed + 1)
        u = torch.rand(f.shape, generator=gen, device=DEV)
        f = torch.where(u < 0.125, torch.zeros_like(f), torch.where(u < 0.25, torch.ones_like(f), f))
        s["f"] = f.contiguous()
    else:
        s["cost"] = _volume(case, seed)
    return s


# -------------------------------------------------------------------- pass --
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "chains":
        return chain_prox(s["y"], w=s.get("w"), lam=case["lam"], out=s["x"])
    if kind == "ragged":
        return chain_prox(s["y"], w=s["w"], offsets=s["offsets"], max_len=s["max_len"], out=s["x"])
    if kind == "backward":
        gy, gw = chain_prox_backward(s["x"], s["grad"], with_w=case["edges"])
        return [gy, gw] if case["edges"] else [gy]
    if kind == "rof":
        x, iters, _, ok = tv2d_denoise(s["f"], lam=case["lam"], w_h=s["wh"], w_v=s["wv"],
                                       max_iters=MAX_ITERS, tol=TOL)
        return [x, iters, ok]
    if kind == "batch":
        xs, iters, _, ok = tv2d_denoise_batched(s["fs"], s["lams"], w_hs=s["whs"], w_vs=s["wvs"],
                                                max_iters=MAX_ITERS, tol=TOL)
        # the images of a batch are one output: at most a few dozen tensors are compared
        return [torch.cat([x.reshape(-1) for x in xs]), np.array(iters), ok]
    if kind == "warm":
        x, iters, _, ok, fallback = learned.denoise_warm(s["net"], s["f"], case["lam"], s["lam_t"],
                                                         tol=TOL, max_iters=MAX_ITERS)
        return [x, iters, ok, fallback]
    if kind == "train":
        net = s["net"]
        net.grad.zero_()
        loss = net.loss_and_grad(s["f"], s["lam"], s["target"])
        return [loss, net.grad]
    if kind == "l1":
        x, iters, _, ok = tv2d_denoise_l1(s["f"], lam=case["lam"], max_iters=case["iters"])
        return [x, iters, ok]
    x, energy = chain_prox_nonconvex(s["cost"], sl=-1.0, sr=1.0, w=STEREO_W, C=STEREO_C)
    return [x, energy]


def work(case):
    """Inputs read once, outputs written once; floating-point operations at the order of the
    linear-time algorithm (about ten per node and chain solve)."""
    kind = case["kind"]
    if kind == "chains":
        n = case["chains"] * case["nodes"]
        return {"bytes": (12 if case["edges"] else 8) * n, "flops": 10 * n}
    if kind == "ragged":
        n = int(_lengths(case).sum())
        return {"bytes": 12 * n + 8 * case["chains"], "flops": 10 * n}
    if kind == "backward":
        n = case["chains"] * case["nodes"]
        return {"bytes": (16 if case["edges"] else 12) * n, "flops": 4 * n}
    if kind in ("rof", "warm"):
        n = case["height"] * case["width"]
        flops = 5 * 2 * 12 * n
        if kind == "warm":  # the network: 3x3 convolutions, 2 -> 32 -> 32 -> 32 -> 1 channels
            flops = 3 * 2 * 12 * n + 2 * 9 * n * (2 * 32 + 32 * 32 + 32 * 32 + 32)
        return {"bytes": (16 if case.get("edges") else 8) * n, "flops": flops}
    if kind == "batch":
        sizes, _ = synth.uneven_image_sizes(case["images"], case["size_seed"])
        n = sum(h * w for h, w in sizes)
        return {"bytes": (16 if case["edges"] else 8) * n, "flops": 6 * 2 * 12 * n}
    if kind == "train":
        n = case["images"] * case["height"] * case["width"]
        return {"bytes": 8 * n, "flops": 3 * 2 * 9 * n * (2 * 32 + 32 * 32 + 32 * 32 + 32)}
    if kind == "l1":
        n = case["height"] * case["width"]
        return {"bytes": 8 * n, "flops": case["iters"] * 2 * 15 * n}
    n = case["rows"] * case["nodes"]
    return {"bytes": (4 * case["labels"] + 4) * n, "flops": 10 * case["labels"] * n}


# ------------------------------------------------------------------- exact --
def _chains64(y, w, ends=None):
    """float64 TV-l2 solution of the columns of y (n, B); w (n, B) edge weights (row i: the edge
    to row i + 1; row n - 1 unused), ends (n, B) True at a chain's last node.

    Splitting by thresholds: a run of nodes with known flows at its two ends is compared with its
    own mean z; the flow m_i = clip(m_{i-1} + z - y_i, -w_i, w_i) of the one-threshold problem
    says which nodes of the minimiser lie above z and which below, the run is cut between them
    (the flow there is +-w), and a run that is not cut is constant at its mean."""
    n, B = y.shape
    lo, hi = -w, w.clone()
    cut = torch.zeros((n, B), dtype=torch.bool, device=y.device)
    cut[-1] = True
    if ends is not None:
        cut |= ends
    lo[cut] = 0.0
    hi[cut] = 0.0
    col = torch.arange(B, device=y.device)
    while True:
        seg = cut.long().cumsum(0) - cut.long()
        base = seg.max(0).values + 1
        idx = seg + (base.cumsum(0) - base)[None, :]
        flow = torch.where(cut, lo, torch.zeros_like(lo))
        into = torch.zeros_like(flow)
        into[1:] = flow[:-1]
        total = int(base.sum())
        num = torch.zeros(total, dtype=y.dtype, device=y.device)
        den = torch.zeros_like(num)
        num.index_add_(0, idx.reshape(-1), (y + flow - into).reshape(-1))
        den.index_add_(0, idx.reshape(-1), torch.ones_like(y).reshape(-1))
        z = (num / den)[idx]
        d = z - y
        side = torch.zeros((n, B), dtype=torch.int8, device=y.device)
        m = torch.zeros(B, dtype=y.dtype, device=y.device)
        for i in range(n):
            t = m + d[i]
            m = torch.minimum(torch.maximum(t, lo[i]), hi[i])
            side[i] = (t < lo[i]).to(torch.int8) - (t > hi[i]).to(torch.int8)
        last = torch.zeros(B, dtype=torch.int8, device=y.device)
        for i in range(n - 1, -1, -1):
            s = side[i]
            keep = (s == 0) & ~cut[i]
            last = torch.where(keep, last, s)
            side[i] = last
        new = torch.zeros_like(cut)
        new[:-1] = (side[:-1] != side[1:]) & ~cut[:-1] & (side[:-1] != 0) & (side[1:] != 0)
        if not bool(new.any()):
            return z
        up = new.clone()
        up[:-1] &= side[1:] > side[:-1]
        u = torch.where(up, w, -w)
        lo = torch.where(new, u, lo)
        hi = torch.where(new, u, hi)
        cut |= new


def _rof64(f, lam, wh, wv, y0, tol, max_iters):
    """The accelerated primal-dual iteration in float64 from the dual y0."""
    H, W = f.shape
    f = f.double()
    full = lambda v, shape: torch.full(shape, float(np.float32(lam)), dtype=torch.float64,
                                       device=f.device) if v is None else v.double()
    wh = torch.nn.functional.pad(full(wh, (H, W - 1)), (0, 1)).t().contiguous()   # (W, H)
    wv = torch.nn.functional.pad(full(wv, (H - 1, W)), (0, 0, 0, 1))
    y = torch.zeros_like(f) if y0 is None else y0.double()
    rows = lambda c, s: _chains64(c.t().contiguous(), s * wh).t().contiguous()
    x = rows(f - y, 1.0)
    xold, tau, sigma, theta = x, 1.0, 1.0, 0.0
    for k in range(max_iters):
        c = y / sigma + x + theta * (x - xold)
        y = sigma * (c - _chains64(c, wv / sigma))
        xn = rows((x + tau * (f - y)) / (1 + tau), tau / (1 + tau))
        tv = (wh[:-1].t() * (xn[:, 1:] - xn[:, :-1]).abs()).sum() + \
            (wv[:-1] * (xn[1:] - xn[:-1]).abs()).sum()
        gap = 0.5 * (xn - f).square().sum() + tv - 0.5 * f.square().sum() + \
            0.5 * (xn + (xn - x) / tau).square().sum()
        xold, x = x, xn
        if float(gap) / (H * W) <= tol:
            return x, k + 1, True
        theta = 1 / math.sqrt(1 + 2 * tau)
        tau, sigma = tau * theta, sigma / theta
    return x, max_iters, False


def _net64(net, f, lam, params):
    """The network's pre-activation o and its dual in float64 (weights and biases ``params``)."""
    B, H, W = f.shape
    x = torch.zeros((B, 16, H, W), dtype=torch.float64, device=f.device)
    x[:, 0] = f.bfloat16().double()
    x[:, 1] = lam.bfloat16().double()[:, None, None]
    for (w, b), (_, _, relu) in zip(params, learned.LAYERS):
        x = torch.nn.functional.conv2d(x, w.permute(0, 3, 1, 2), b, padding=1)
        x = torch.relu(x) if relu else x
    p = lam.double()[:, None, None] * torch.tanh(x[:, 0])
    p = torch.cat([p[:, :-1], torch.zeros_like(p[:, :1])], 1)
    return torch.cat([-p[:, :1], p[:, :-1] - p[:, 1:]], 1)


def _params64(net):
    out = []
    for (cin, cout, _), (wo, bo) in zip(learned.LAYERS, net.offsets):
        out.append((net.params_bf16[wo:wo + cout * 9 * cin].view(cout, 3, 3, cin).double(),
                    net.params[bo:bo + cout].double()))
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "l1" or kind == "batch":
        return None   # minutes in float64 torch
    s = prepare(case, seed)
    if kind == "chains":
        w = s["w"].double() if case["edges"] else torch.full_like(s["y"], float(np.float32(case["lam"])),
                                                                  dtype=torch.float64)
        return _chains64(s["y"].double().t().contiguous(), w.t().contiguous()).t().contiguous()
    if kind == "ragged":
        B, n = case["chains"], s["max_len"]
        off = s["offsets"]
        pos = off[:-1][None, :] + torch.arange(n, device=DEV)[:, None]
        ok = pos < off[1:][None, :]
        pos = torch.where(ok, pos, torch.zeros_like(pos))
        y = torch.where(ok, s["y"][pos].double(), torch.zeros((), dtype=torch.float64, device=DEV))
        w = torch.where(ok, s["w"][pos].double(), torch.zeros((), dtype=torch.float64, device=DEV))
        ends = torch.zeros_like(ok)
        ends[:-1] = ok[:-1] & ~ok[1:]
        z = _chains64(y, w, ends)
        return z.t()[ok.t()].contiguous()
    if kind == "backward":
        x, g = s["x"], s["grad"].double()
        B, n = x.shape
        head = torch.ones_like(x, dtype=torch.bool)
        head[:, 1:] = x[:, 1:] != x[:, :-1]
        seg = head.reshape(-1).long().cumsum(0) - 1
        total = int(seg[-1]) + 1
        num = torch.zeros(total, dtype=torch.float64, device=DEV).index_add_(0, seg, g.reshape(-1))
        den = torch.zeros_like(num).index_add_(0, seg, torch.ones_like(g).reshape(-1))
        gy = (num / den)[seg].view(B, n)
        if not case["edges"]:
            return [gy]
        gw = torch.zeros_like(gy)
        gw[:, :-1] = torch.sign(x[:, 1:] - x[:, :-1]).double() * (gy[:, :-1] - gy[:, 1:])
        return [gy, gw]
    if kind == "rof":
        return list(_rof64(s["f"], case["lam"], s["wh"], s["wv"], None, TOL, MAX_ITERS))
    if kind == "warm":
        with torch.no_grad():
            y0 = _net64(s["net"], s["f"][None], s["lam_t"], _params64(s["net"]))[0]
        x, iters, ok = _rof64(s["f"], case["lam"], None, None, y0, TOL, 6)
        return [x, None, None, None] if ok else None
    if kind == "train":
        net = s["net"]
        params = [(w.requires_grad_(True), b.requires_grad_(True)) for w, b in _params64(net)]
        loss = (_net64(net, s["f"], s["lam"], params) - s["target"].double()).square().mean()
        loss.backward()
        grad = torch.zeros(net.numel, dtype=torch.float64, device=DEV)
        for (w, b), (wo, bo) in zip(params, net.offsets):
            grad[wo:wo + w.numel()] = w.grad.reshape(-1)
            grad[bo:bo + b.numel()] = b.grad
        return [loss.detach().reshape(1), grad]
    # the integers hold a minimiser: breakpoints at 0 .. labels - 1, C / w a whole number
    cost = s["cost"]
    R, n, L = cost.shape
    reach = int(STEREO_C / STEREO_W)
    lab = torch.arange(-reach, reach + 1, device=DEV).abs().double() * STEREO_W
    m = cost[:, 0].double()
    for i in range(1, n):
        far = m.min(1, keepdim=True).values + STEREO_C
        pad = torch.nn.functional.pad(m, (reach, reach), value=float("inf"))
        near = (pad.unfold(1, 2 * reach + 1, 1) + lab).min(2).values
        m = torch.minimum(near, far) + cost[:, i].double()
    return [None, m.min(1).values]
