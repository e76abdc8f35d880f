"""Workloads of the stereo matcher: what a program that uses this package has it do.

Every case goes through the package's public entry points (the C ABI's Python binding and
the proposal network's training class) on synthetic rectified pairs shaped like the
package's own scenes: a four-octave gradient-noise texture, slanted planes on Voronoi
regions, a z-buffered right view and sensor noise.  The texture and the warp run on the
GPU so that inputs are quick to make.

Kinds
  match     one pair on the device, mpv_match (summed merge, pyramid windows); with merge,
            gradient or learned set: the layered merge, the gradient-weighted penalty or
            the learned window proposal
  host      one pair in pinned host buffers, mpv_match_host
  batch     pairs of mixed sizes in one mpv_match_batch call
  road      v/u-disparity and road profile of a disparity map, mpv_road_detect
  train     forward, loss and gradients of the proposal network, learn.Net
"""
import math
import os

import numpy as np
import torch
import torch.nn.functional as F

from paper_2001_09678_gb300 import learn, mpv

DEV = "cuda"
WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(learn.__file__)), "weights",
                       "proposal_d128_s3.bin")


def _match(name, w, h, d, scales=3, paths=8, n=5, lr=1, merge=0, gradient=False, learned=0):
    return dict(name=name, kind="match", w=w, h=h, d=d, scales=scales, paths=paths, n=n, lr=lr,
                merge=merge, gradient=gradient, learned=learned)


def listed():
    return [
        # the smallest call: a 320x240 frame of one scale and 4 paths, where latency counts
        _match("qvga_1scale_4path", 320, 240, 32, scales=1, paths=4),
        # a VGA camera whose frames live in host memory (copies in and out inside the call)
        dict(name="vga_host", kind="host", w=640, h=480, d=64, scales=3, paths=8, n=5, lr=1),
        # the ordinary frame: 1280x720, 128 labels, three scales, both views
        _match("hd", 1280, 720, 128),
        # the largest camera of the served streams
        _match("fhd", 1920, 1080, 192),
        # odd sizes: rows, labels and windows (25 labels) that fill no tile or stride
        _match("ragged", 1237, 371, 100),
        # the exact method at full range (one scale): the judge and the fallback of the
        # learned proposal, and the choice of callers who want no pyramid
        _match("hd_full_range", 1280, 720, 128, scales=1),
        # the layered path merge of the method's own paper
        _match("hd_layered", 1280, 720, 128, merge=1),
        # the gradient-weighted jump penalty
        _match("hd_gradient", 1280, 720, 128, gradient=True),
        # windows from the learned proposal (network on the tensor cores, 17 labels)
        _match("hd_learned", 1280, 720, 128, learned=17),
        # pairs of mixed sizes and ranges in one submission, as a multi-camera rig has them
        dict(name="batch_mixed", kind="batch", vga=3, hd=6, fhd=3),
        # the road profile on a frame's disparity map
        dict(name="road_hd", kind="road", w=1280, h=720, d=128, eta=8),
        # one training step's forward pass, loss and gradients at the training batch size
        dict(name="train", kind="train", batch=8, cin=34, w=320, h=180),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["match", "match", "match", "full", "merge", "gradient", "learned", "host",
                       "batch", "road", "train"])
    if kind == "train":
        return dict(kind="train", batch=rng.randint(1, 8), cin=34, w=_log_int(rng, 40, 320),
                    h=_log_int(rng, 24, 180))
    if kind == "batch":
        return dict(kind="batch", vga=rng.randint(0, 4), hd=rng.randint(1, 5), fhd=rng.randint(0, 2))
    if kind == "road":
        return dict(kind="road", w=_log_int(rng, 320, 1920), h=_log_int(rng, 200, 1080),
                    d=_log_int(rng, 32, 192), eta=rng.randint(4, 16))
    if kind in ("learned", "gradient", "merge"):
        w, h = _log_int(rng, 480, 1280), _log_int(rng, 270, 720)
    elif kind == "full":
        w, h = _log_int(rng, 320, 1280), _log_int(rng, 180, 720)
    else:
        w, h = _log_int(rng, 320, 1920), _log_int(rng, 200, 1080)
    d = 128 if kind == "learned" else min(_log_int(rng, 32, 128 if kind == "full" else 192), w // 2)
    c = _match(None, w, h, d, scales=1 if kind == "full" else (3 if kind == "learned" else
               rng.choice([2, 3, 3])), paths=rng.choice([4, 8, 8]), n=rng.choice([3, 5, 5]),
               lr=1 if kind == "learned" else rng.choice([0, 1, 1, 1]),
               merge=int(kind == "merge"), gradient=kind == "gradient",
               learned=rng.choice([16, 17]) if kind == "learned" else 0)
    del c["name"]
    if kind == "host":
        c = dict(kind="host", w=w, h=h, d=d, scales=c["scales"], paths=c["paths"], n=c["n"],
                 lr=c["lr"])
    return c


# ---------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------

def _texture(gen, w, h, octaves=4, period=64.0, contrast=110.0):
    """Gradient noise (quintic fade, 16 directions), four octaves, uint8 [h][w]."""
    acc = torch.zeros(h, w, device=DEV)
    for o in range(octaves):
        p = period / 2 ** o
        gh, gw = int(h / p) + 3, int(w / p) + 3
        a = torch.randint(0, 16, (gh, gw), generator=gen, device=DEV) * (2 * math.pi / 16)
        gx, gy = torch.cos(a), torch.sin(a)
        y = (torch.arange(h, device=DEV) + 0.5) / p
        x = (torch.arange(w, device=DEV) + 0.5) / p
        yi, xi = y.long(), x.long()
        yf, xf = (y - yi)[:, None], (x - xi)[None, :]

        def dot(dy, dx):
            iy, ix = (yi + dy)[:, None], (xi + dx)[None, :]
            return gx[iy, ix] * (xf - dx) + gy[iy, ix] * (yf - dy)

        u = xf * xf * xf * (xf * (xf * 6 - 15) + 10)
        v = yf * yf * yf * (yf * (yf * 6 - 15) + 10)
        top = dot(0, 0) * (1 - u) + dot(0, 1) * u
        bot = dot(1, 0) * (1 - u) + dot(1, 1) * u
        acc += 0.5 ** o * 1.41421356 * (top * (1 - v) + bot * v)
    scale = sum(0.5 ** o for o in range(octaves))
    return torch.clamp(torch.round(128 + contrast * 2 * acc / scale), 0, 255).to(torch.int64)


def _planes(gen, w, h, d_max, n=40, slope=0.2):
    """Disparity of slanted planes on the Voronoi regions of n random seeds, [h][w]."""
    r = torch.rand(n, 5, generator=gen, device=DEV)
    sx, sy, d0 = r[:, 0] * w, r[:, 1] * h, r[:, 2] * d_max
    gx, gy = (r[:, 3] * 2 - 1) * slope, (r[:, 4] * 2 - 1) * slope
    y = torch.arange(h, device=DEV, dtype=torch.float32)[:, None]
    x = torch.arange(w, device=DEV, dtype=torch.float32)[None, :]
    best = torch.full((h, w), 1e30, device=DEV)
    disp = torch.zeros(h, w, device=DEV)
    for k in range(n):
        q = (x - sx[k]) ** 2 + (y - sy[k]) ** 2
        near = q < best
        best = torch.where(near, q, best)
        disp = torch.where(near, d0[k] + gx[k] * (x - sx[k]) + gy[k] * (y - sy[k]), disp)
    return disp.clamp(0, d_max)


def _pair(seed, w, h, d):
    """A rectified pair: uint8 left and right images on the device."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    left = _texture(gen, w, h)
    holes = _texture(gen, w, h)
    disp = _planes(gen, w, h, 0.94 * (d - 1))
    x = torch.arange(w, device=DEV)[None, :]
    to = x - torch.round(disp).long()
    row = torch.arange(h, device=DEV)[:, None] * w
    key = (torch.round(disp * 16).long() << 8) | left
    ok = to >= 0
    z = torch.full((h * w,), -1, dtype=torch.int64, device=DEV)
    z.scatter_reduce_(0, (row + to)[ok], key[ok], reduce="amax")
    z = z.view(h, w)
    right = torch.where(z >= 0, z & 255, holes).float()
    right = right + 2.0 * torch.randn(h, w, generator=gen, device=DEV)
    return left.to(torch.uint8), torch.clamp(torch.round(right), 0, 255).to(torch.uint8)


def _gradient_table(p1=10, sigma=16.0):
    g = np.arange(256, dtype=np.float64)
    return np.floor(p1 * np.exp(-g / sigma) + 0.5).astype(np.int32)


class _Ctx:
    """A matcher context that is released with the state that holds it."""

    def __init__(self, **params):
        self.h = mpv.mpv_create(0)
        mpv.mpv_set_params(self.h, mpv.mpv_default_params(**params))

    def __del__(self):
        if mpv is not None:
            mpv.mpv_destroy(self.h)


def _params(c):
    p = dict(max_disparity=c["d"], num_scales=c["scales"], num_paths=c["paths"], p1=10, trunc=30,
             ssim_window=c["n"], lr_check=c["lr"], lr_tol=1)
    if c.get("merge"):
        p["merge_mode"] = mpv.MPV_MERGE_PAPER
    if c.get("learned"):
        p.update(proposal=mpv.MPV_PROPOSAL_LEARNED, window=c["learned"])
    return p


def prepare(case, seed):
    kind = case["kind"]
    mpv.load()
    if kind == "train":
        gen = torch.Generator(device=DEV).manual_seed(seed)
        b, cin, h, w = case["batch"], case["cin"], case["h"], case["w"]
        # network input: two images in [-1/2, 1/2] and matching costs in [0, 1]
        x = torch.rand(b, cin, h, w, generator=gen, device=DEV)
        x[:, :2] -= 0.5
        target = F.interpolate(torch.rand(b, 1, 6, 8, generator=gen, device=DEV), size=(h, w),
                               mode="bilinear")
        return dict(kind=kind, net=learn.Net(learn.init_weights(cin, seed)),
                    x=x.to(torch.bfloat16), target=target.contiguous())
    if kind == "road":
        gen = torch.Generator(device=DEV).manual_seed(seed)
        w, h, d = case["w"], case["h"], case["d"]
        # a flat road below the horizon, obstacles in front of it, and rejected pixels
        y = torch.arange(h, device=DEV, dtype=torch.float32)[:, None]
        road = ((y - 0.35 * h).clamp(min=0) / (0.65 * h) * 0.9 * (d - 1)).expand(h, w)
        m = torch.maximum(road, _planes(gen, w, h, 0.5 * d) * (torch.rand(
            h // 32 + 1, w // 32 + 1, generator=gen, device=DEV) < 0.3).repeat_interleave(
                32, 0)[:h].repeat_interleave(32, 1)[:, :w])
        m = torch.round(m + 0.4 * torch.randn(h, w, generator=gen, device=DEV)).clamp(0, d - 1)
        m = torch.where(torch.rand(h, w, generator=gen, device=DEV) < 0.12,
                        torch.full_like(m, -1.0), m)     # 0xFFFF: rejected by the check
        i32 = dict(dtype=torch.int32, device=DEV)
        return dict(kind=kind, ctx=_Ctx(max_disparity=d), disp=m.to(torch.int16).contiguous(), d=d,
                    eta=case["eta"], vdisp=torch.empty(h, d, **i32), udisp=torch.empty(w, d, **i32),
                    profile=torch.empty(d, **i32),
                    energy=torch.empty(1, dtype=torch.int64, device=DEV))
    if kind == "batch":
        shapes = ([(640, 480, 64)] * case["vga"] + [(1280, 720, 128)] * case["hd"] +
                  [(1920, 1080, 192)] * case["fhd"])
        ctx = _Ctx(max_disparity=128)
        pairs = []
        for i, (w, h, d) in enumerate(shapes):
            left, right = _pair(seed * 64 + i, w, h, d)
            pairs.append(dict(left=left, right=right, max_disparity=d,
                              disp=torch.empty(h, w, dtype=torch.int16, device=DEV)))
        mpv.mpv_match_batch(ctx.h, pairs)     # tunes the launch shapes once per set of sizes
        mpv.mpv_sync(ctx.h)
        return dict(kind=kind, ctx=ctx, pairs=pairs)
    left, right = _pair(seed, case["w"], case["h"], case["d"])
    ctx = _Ctx(**_params(case))
    if case.get("gradient"):
        mpv.mpv_set_gradient_penalty(ctx.h, _gradient_table())
    if case.get("learned"):
        mpv.mpv_load_proposal_weights(ctx.h, WEIGHTS)
    shape = (case["h"], case["w"])
    if kind == "host":
        return dict(kind=kind, ctx=ctx, left=left.cpu().pin_memory(), right=right.cpu().pin_memory(),
                    disp=torch.empty(shape, dtype=torch.int16).pin_memory())
    return dict(kind=kind, ctx=ctx, left=left, right=right,
                disp=torch.empty(shape, dtype=torch.int16, device=DEV))


def run(state):
    kind = state["kind"]
    if kind == "match":
        mpv.mpv_match(state["ctx"].h, state["left"], state["right"], state["disp"])
        return state["disp"]
    if kind == "host":
        mpv.mpv_match_host(state["ctx"].h, state["left"], state["right"], state["disp"])
        return state["disp"]
    if kind == "batch":
        mpv.mpv_match_batch(state["ctx"].h, state["pairs"])
        return [q["disp"] for q in state["pairs"]]
    if kind == "road":
        mpv.mpv_road_detect(state["ctx"].h, state["disp"], state["d"], state["eta"], state["vdisp"],
                            state["profile"], state["energy"], state["udisp"])
        return dict(vdisp=state["vdisp"], udisp=state["udisp"], profile=state["profile"],
                    energy=state["energy"])
    net = state["net"]
    pred, acts = net.forward(state["x"])
    grad = torch.empty_like(pred)
    loss = torch.zeros(1, dtype=torch.float32, device=DEV)
    mpv.mpv_cnn_huber(pred, state["target"], 1.0 / 128, grad, loss)
    grads = net.backward(acts, grad)
    return dict(pred=pred, loss=loss, dw=[g[0] for g in grads], db=[g[1] for g in grads])


# ---------------------------------------------------------------------------------------
# Work of one pass, and outputs in 64 bits
# ---------------------------------------------------------------------------------------

def _nodes(c):
    """Evaluated (pixel, label) nodes of one view and of the levels that are aggregated."""
    levels, w, h = [], c["w"], c["h"]
    s = c["scales"]
    for l in range(s - 1, -1, -1):
        full = (c["d"] + (1 << (s - 1 - l)) - 1) >> (s - 1 - l)
        win = full if l == 0 else min(max(c["d"] // 4, 1), full)
        if c.get("learned") and l == s - 1:
            win = c["learned"]
        levels.append(w * h * win)
        w, h = (w + 1) // 2, (h + 1) // 2
    if c.get("learned"):          # the top level's costs feed the network, no level between
        return levels[0] + levels[-1], levels[0]
    return sum(levels), sum(levels)


def work(case):
    kind = case["kind"]
    if kind == "train":
        px = case["batch"] * case["w"] * case["h"]
        shapes = learn.layer_shapes(case["cin"])
        macs = sum(9 * ci * co for ci, co, _ in shapes)
        back = sum(9 * ci * co for ci, co, _ in shapes[1:])
        par = sum(9 * ci * co + co for ci, co, _ in shapes)
        return {"bytes": px * (2 * case["cin"] + 8) + par * 10, "flops": 2 * px * (2 * macs + back)}
    if kind == "road":
        w, h, d = case["w"], case["h"], case["d"]
        return {"bytes": 2 * w * h + 4 * d * (w + h + 1) + 8, "flops": 2 * w * h + h * d * case["eta"]}
    if kind == "batch":
        total = {"bytes": 0, "flops": 0}
        for count, (w, h, d) in ((case["vga"], (640, 480, 64)), (case["hd"], (1280, 720, 128)),
                                 (case["fhd"], (1920, 1080, 192))):
            one = work(_match("", w, h, d))
            for k in total:
                total[k] += count * one[k]
        return total
    views = 2 if case["lr"] else 1
    cost, agg = _nodes(case)
    # two images in, one 16-bit map out.  Operations of a node: the sliding column products
    # (2 N) and the quotient (12) of its cost; per direction four neighbours' add and min, the
    # cap, the path's minimum and the sum (12)
    flops = views * (cost * (2 * case["n"] + 12) + agg * case["paths"] * 12)
    if case.get("learned"):
        macs = sum(9 * ci * co for ci, co, _ in learn.layer_shapes(2 + case["d"] // 4))
        flops += views * 2 * macs * (case["w"] // 4) * (case["h"] // 4)
    return {"bytes": 4 * case["w"] * case["h"], "flops": flops}


def _bf16(t):
    return t.float().to(torch.bfloat16).double()


def exact(case, seed):
    """Training: the network in 64 bits, its weights and stored activations BF16 as the network
    defines them.  The matcher and the road profile return whole numbers."""
    if case["kind"] != "train":
        return None
    st = prepare(case, seed)
    layers = st["net"].layers
    acts = [st["x"].double()]
    for i, l in enumerate(layers):
        h = F.conv2d(acts[-1], l["wb"].double(), l["b"].double(), padding=1)
        acts.append(_bf16(h.clamp(min=0)) if i + 1 < len(layers) else h)
    pred, delta = acts[-1], 1.0 / 128
    r = pred - st["target"].double()
    a = r.abs()
    loss = torch.where(a < delta, 0.5 * r * r / delta, a - 0.5 * delta).mean().reshape(1)
    g = torch.where(a < delta, r / delta, torch.sign(r)) / r.numel()
    dw, db = [None] * len(layers), [None] * len(layers)
    for i in range(len(layers) - 1, -1, -1):
        w = layers[i]["wb"].double()
        if layers[i]["relu"]:
            g = g * (acts[i + 1] > 0)
        db[i] = g.sum((0, 2, 3))
        dw[i] = torch.nn.grad.conv2d_weight(acts[i], w.shape, g, padding=1)
        if i:
            g = F.conv_transpose2d(g, w, padding=1)
    return dict(pred=pred, loss=loss, dw=dw, db=db)
