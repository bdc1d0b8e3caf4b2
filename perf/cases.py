"""The work this package is asked to do, as measurable cases.

ExWarp inserts frames P_1..P_3 between two rendered frames by warping the last one with its motion vectors.  The
cases below are the calls a renderer, a streaming host and a trainer make through the public entry points, over the
range of sizes, colour types and scenes they meet.  Scenes are drawn on the GPU from a seed: value-noise surfaces, a
background plane at depth 100 under a camera pan (or a dolly with roll, whose motion varies from pixel to pixel), and
rectangles of random depth with a velocity of their own; what they uncover are the holes.

``exact`` computes the same outputs in 64-bit floating point with plain torch.
"""
import math

import numpy as np
import torch

from paper_2307_12607_gb300 import autograd, binding

DT = {"f32": torch.float32, "f16": torch.float16}
CDT = {"f32": binding.F32, "f16": binding.F16}


def _dev():
    return torch.device("cuda", torch.cuda.current_device())


# ---------------------------------------------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------------------------------------------

def listed():
    return [
        # One low-resolution frame on its own: the smallest call, what a game adds between two rendered frames.
        {"name": "frame_360p_f32", "kind": "frames", "W": 640, "H": 360, "frames": 1, "dtype": "f32", "fill": True,
         "objects": 8, "vmax": 12.0, "camera": "pan"},
        # The paper's 480p (854 x 480): rows that are not a multiple of 16 bytes.
        {"name": "frame_480p_f32", "kind": "frames", "W": 854, "H": 480, "frames": 1, "dtype": "f32", "fill": True,
         "objects": 16, "vmax": 12.0, "camera": "pan"},
        # A camera that moves and turns: motion differs from pixel to pixel everywhere (a few frames, FP16 colour).
        {"name": "dolly_1080p_f16", "kind": "frames", "W": 1920, "H": 1080, "frames": 4, "dtype": "f16", "fill": True,
         "objects": 32, "vmax": 12.0, "camera": "dolly"},
        # The benchmark's sequence: 60 source frames, 180 inserted ones.
        {"name": "sequence_1080p_f32", "kind": "frames", "W": 1920, "H": 1080, "frames": 60, "dtype": "f32",
         "fill": True, "objects": 32, "vmax": 12.0, "camera": "pan"},
        # One 4K frame with fast nearby occluders, warp and mask only (the caller fills with a network of its own).
        {"name": "warp_4k_f16", "kind": "frames", "W": 3840, "H": 2160, "frames": 1, "dtype": "f16", "fill": False,
         "objects": 68, "vmax": 48.0, "camera": "pan"},
        # A streaming host: 48 independent streams of four resolutions in one call.
        {"name": "batched_48_streams", "kind": "batched", "W": 3840, "H": 2160, "streams": 48, "dtype": "f16",
         "objects": 40, "vmax": 12.0, "camera": "pan"},
        # Training through the warp: forward, L2 loss and gradients of eight frames, all three fractions.
        {"name": "train_1080p_f32", "kind": "train", "W": 1920, "H": 1080, "frames": 8, "dtype": "f32", "objects": 32,
         "vmax": 12.0, "camera": "pan"},
        # The same from torch, one fraction with a loss of the user's own: the warp under autograd, back and forth.
        {"name": "autograd_720p_f32", "kind": "autograd", "W": 1280, "H": 720, "dtype": "f32", "k": 2, "objects": 24,
         "vmax": 12.0, "camera": "pan"},
        # Frames warped from warped frames (decision path S6): three quarter steps.
        {"name": "recursive_1080p_f32", "kind": "recursive", "W": 1920, "H": 1080, "steps": 3, "dtype": "f32",
         "objects": 32, "vmax": 12.0, "camera": "pan"},
        # The stages one by one for one fraction, FP16: splat, warp, fill.
        {"name": "staged_720p_f16", "kind": "staged", "W": 1280, "H": 720, "dtype": "f16", "k": 3, "objects": 24,
         "vmax": 12.0, "camera": "pan"},
        # The decision stage's motion features of a frame.
        {"name": "features_1080p", "kind": "features", "W": 1920, "H": 1080, "dtype": "f32", "objects": 32,
         "vmax": 12.0, "camera": "dolly"},
        # The reward of an inserted frame against the rendered one: PSNR and SSIM.
        {"name": "reward_1080p_f32", "kind": "reward", "W": 1920, "H": 1080, "dtype": "f32", "objects": 32,
         "vmax": 12.0, "camera": "pan"},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, wlo, whi):
    """A width over the range on a log scale, a 16:9-like height; as often as not a common multiple of 16."""
    W = _logint(rng, wlo, whi)
    H = max(160, int(W * rng.uniform(0.5, 0.7)))
    if rng.random() < 0.5:
        W, H = W // 16 * 16, H // 8 * 8
    return W, H


def draw(rng):
    kind = rng.choice(["frames", "frames", "frames", "batched", "train", "autograd", "recursive", "staged",
                       "features", "reward"])
    c = {"kind": kind, "dtype": rng.choice(["f32", "f16"]), "camera": rng.choice(["pan", "pan", "dolly"])}
    if kind == "batched":
        c["W"], c["H"] = _size(rng, 960, 2560)
        c["streams"] = rng.randint(4, 24)
    elif kind == "train":
        c["W"], c["H"] = _size(rng, 480, 1920)
        c["frames"] = rng.randint(1, 8)
    else:
        c["W"], c["H"] = _size(rng, 360, 3840)
    if kind == "frames":
        c["frames"] = max(1, min(_logint(rng, 1, 60), int(60 * 1920 * 1080 * 0.4 / (c["W"] * c["H"]))))
        c["fill"] = rng.random() < 0.7
    if kind in ("autograd", "staged"):
        c["k"] = rng.randint(1, 3)
    if kind == "recursive":
        c["steps"] = rng.randint(2, 3)
    c["objects"] = rng.randint(8, 64)
    c["vmax"] = 48.0 if c["W"] > 2600 and rng.random() < 0.5 else 12.0
    return c


def _stream_sizes(case):
    """Equal shares of four resolutions: 1/3, 1/2, 2/3 and all of the largest."""
    W, H, n = case["W"], case["H"], case["streams"]
    shares = ((1, 3), (1, 2), (2, 3), (1, 1))
    groups = {}
    for s in range(n):
        a, b = shares[s * 4 // n]
        groups.setdefault((W * a // b, H * a // b), []).append(s)
    return groups


def work(case):
    px = case["W"] * case["H"]
    c = 6 if case["dtype"] == "f16" else 12
    kind = case["kind"]
    # a gathered pixel: three channels of a four-tap bilinear sum and one scaling, the weights, the splat's compares
    per_out = 3 * 8 + 30
    if kind == "frames":  # the source once, three colours and masks written
        return {"bytes": case["frames"] * px * ((c + 12) + 3 * (c + 1)), "flops": case["frames"] * px * 3 * per_out}
    if kind == "batched":
        n = sum(w * h * len(s) for (w, h), s in _stream_sizes(case).items())
        return {"bytes": n * ((c + 12) + 3 * (c + 1)), "flops": n * 3 * per_out}
    if kind == "train":  # the source and three targets read, five gradient planes written
        return {"bytes": case["frames"] * px * ((c + 12) + 3 * c + 20), "flops": case["frames"] * px * 3 * 3 * per_out}
    if kind == "autograd":  # forward: source in, colour and mask out; backward: gradient in, two gradients out
        return {"bytes": px * ((c + 12) + (c + 1) + (c + 12) + c + c + 8), "flops": px * 4 * per_out}
    if kind == "recursive":  # colour, depth and motion in, a colour and a mask out per step
        return {"bytes": px * ((c + 12) + case["steps"] * (c + 1)), "flops": case["steps"] * px * per_out}
    if kind == "staged":  # source in; keys, mask and filled colour out
        return {"bytes": px * ((c + 12) + 8 + (c + 1)), "flops": px * per_out}
    if kind == "features":
        return {"bytes": px * 8, "flops": px * 6}
    # PSNR and SSIM of one pair of images: each read once; five windowed moments, separable, per value
    return {"bytes": px * 2 * c, "flops": px * 3 * (3 + 5 * 2 * 2 * 11 + 16)}


# ---------------------------------------------------------------------------------------------------------------
# Scenes
# ---------------------------------------------------------------------------------------------------------------
CELL = 8.0      # value-noise lattice pitch in pixels
PERIOD = 64     # cells per period of the background


def _disc(rng, rmax):
    r, th = rmax * math.sqrt(rng.uniform()), rng.uniform(0.0, 2.0 * math.pi)
    return r * math.cos(th), r * math.sin(th)


def _scene(W, H, objects, vmax, camera, rng, dev):
    px, py = _disc(rng, vmax / 3.0)
    s = {"W": W, "H": H, "pan": (float(np.float32(px)), float(np.float32(py))), "dolly": None, "rects": []}
    if camera == "dolly":  # towards the scene by up to 1% a frame, turning by up to half a degree
        s["dolly"] = (float(rng.uniform(0.004, 0.01) * rng.choice([-1.0, 1.0])),
                      float(math.radians(rng.uniform(0.1, 0.5)) * rng.choice([-1.0, 1.0])))
    s["back"] = torch.from_numpy(rng.uniform(0.05, 0.95, size=(3, PERIOD, PERIOD)).astype(np.float32)).to(dev)
    fast = objects // 16 if vmax > 12.0 else 0
    for i in range(objects):
        if i < objects // 20:  # slivers of 1 to 3 pixels
            w, h = float(rng.integers(1, 4)), rng.uniform(H / 8, H / 2)
            if rng.uniform() < 0.5:
                w, h = h, w
        elif i >= objects - fast:  # nearby occluders, each about a twentieth of the frame, at full speed
            w = math.sqrt(0.05 * W * H * rng.uniform(0.5, 2.0))
            h = 0.05 * W * H / w
        else:
            w, h = rng.uniform(W / 24, W / 6), rng.uniform(H / 24, H / 6)
        near = i >= objects - fast
        vx, vy = _disc(rng, vmax)
        depth = rng.uniform(0.1, 0.5) if near else rng.uniform(0.1, 99.0)
        lx, ly = int(math.ceil(w / CELL)) + 2, int(math.ceil(h / CELL)) + 2
        lat = rng.uniform(0.0, 1.0, size=(3, 1, 1)) + rng.uniform(0.2, 0.6) * (rng.uniform(size=(3, ly, lx)) - 0.5)
        s["rects"].append({"x": rng.uniform(-0.5 * w, W - 0.5 * w), "y": rng.uniform(-0.5 * h, H - 0.5 * h), "w": w,
                           "h": h, "v": (float(np.float32(vx + px)), float(np.float32(vy + py))),
                           "depth": float(np.float32(depth)),
                           "lat": torch.from_numpy(np.clip(lat, 0.0, 1.0).astype(np.float32)).to(dev)})
    s["rects"].sort(key=lambda r: -r["depth"])  # painted far to near
    return s


def _noise(lat, u, v, periodic):
    """Value noise of the lattice at columns u and rows v (float64 pixels): [3][len(v)][len(u)]."""
    def axis(t, n):
        t = t / CELL
        i = torch.floor(t)
        f = (t - i).to(torch.float32)
        i = i.to(torch.int64)
        a, b = (i % n, (i + 1) % n) if periodic else (i.clamp(0, n - 1), (i + 1).clamp(0, n - 1))
        return a, b, f * f * (3.0 - 2.0 * f)
    i0, i1, su = axis(u, lat.shape[2])
    j0, j1, sv = axis(v, lat.shape[1])
    cols = lat[:, :, i0] * (1.0 - su) + lat[:, :, i1] * su
    return cols[:, j0, :] * (1.0 - sv)[:, None] + cols[:, j1, :] * sv[:, None]


def _render(s, t, color, depth, mv):
    """Colour, depth and motion of scene s at time t (frames) into the given tensors."""
    W, H, dev = s["W"], s["H"], depth.device
    xs = torch.arange(W, dtype=torch.float64, device=dev)
    ys = torch.arange(H, dtype=torch.float64, device=dev)
    color.copy_(_noise(s["back"], xs - s["pan"][0] * t, ys - s["pan"][1] * t, True))
    depth.fill_(100.0)
    mv[0].fill_(s["pan"][0])
    mv[1].fill_(s["pan"][1])
    if s["dolly"] is not None:
        zoom, turn = s["dolly"]
        x, y = (xs - 0.5 * W).to(torch.float32)[None, :], (ys - 0.5 * H).to(torch.float32)[:, None]
        mv[0].add_(zoom * x - turn * y)
        mv[1].add_(turn * x + zoom * y)
    for r in s["rects"]:
        x0, y0 = r["x"] + r["v"][0] * t, r["y"] + r["v"][1] * t
        xa, xb = max(0, math.ceil(x0)), min(W, math.ceil(x0 + r["w"]))
        ya, yb = max(0, math.ceil(y0)), min(H, math.ceil(y0 + r["h"]))
        if xa >= xb or ya >= yb:
            continue
        color[:, ya:yb, xa:xb] = _noise(r["lat"], xs[xa:xb] - x0, ys[ya:yb] - y0, False).to(color.dtype)
        depth[ya:yb, xa:xb] = r["depth"]
        mv[0, ya:yb, xa:xb] = r["v"][0]
        mv[1, ya:yb, xa:xb] = r["v"][1]


def _buffers(n, W, H, dtype, dev):
    return (torch.empty((n, 3, H, W), dtype=DT[dtype], device=dev),
            torch.empty((n, H, W), dtype=torch.float32, device=dev),
            torch.empty((n, 2, H, W), dtype=torch.float32, device=dev))


def _frames(case, seed, n, W, H, salt=0):
    """n consecutive frames of one scene: (scene, colour [n][3][H][W], depth [n][H][W], motion [n][2][H][W])."""
    dev = _dev()
    rng = np.random.Generator(np.random.PCG64([int(seed), salt]))
    s = _scene(W, H, case["objects"], case["vmax"], case["camera"], rng, dev)
    color, depth, mv = _buffers(n, W, H, case["dtype"], dev)
    for f in range(n):
        _render(s, float(f), color[f], depth[f], mv[f])
    return s, color, depth, mv


def _truth(s, t, dtype, W, H):
    """The scene's colour at time t: what an inserted frame should show."""
    color, depth, mv = _buffers(1, W, H, dtype, _dev())
    _render(s, t, color[0], depth[0], mv[0])
    return color[0]


# ---------------------------------------------------------------------------------------------------------------
# What a program has in hand, and one pass
# ---------------------------------------------------------------------------------------------------------------

def _inputs(case, seed):
    """The inputs alone, shared by prepare and exact."""
    kind, W, H = case["kind"], case["W"], case["H"]
    if kind == "frames":
        return _frames(case, seed, case["frames"], W, H)[1:]
    if kind == "batched":
        groups = []
        for (w, h), members in _stream_sizes(case).items():
            color, depth, mv = _buffers(len(members), w, h, case["dtype"], _dev())
            for i, m in enumerate(members):
                _, c, d, v = _frames(case, seed, 1, w, h, salt=1 + m)
                color[i], depth[i], mv[i] = c[0], d[0], v[0]
            groups.append((color, depth, mv))
        return groups
    if kind == "train":
        s, color, depth, mv = _frames(case, seed, case["frames"], W, H)
        target = torch.empty((case["frames"], 3, 3, H, W), dtype=color.dtype, device=color.device)
        for f in range(case["frames"]):
            for k in range(3):
                target[f, k] = _truth(s, f + 0.25 * (k + 1), case["dtype"], W, H)
        return color, depth, mv, target
    s, color, depth, mv = _frames(case, seed, 1, W, H)
    if kind == "autograd":
        g = torch.Generator(device=color.device).manual_seed(int(seed))
        grad = torch.randn((3, H, W), generator=g, device=color.device).to(color.dtype)
        return color[0], depth[0], mv[0], grad
    if kind == "features":
        return (mv[0],)
    if kind == "reward":  # a frame half a pixel or so off the rendered one, as a warped frame is
        g = torch.Generator(device=color.device).manual_seed(int(seed))
        other = _truth(s, 0.05, "f32", W, H)
        other += 0.004 * torch.randn((3, H, W), generator=g, device=color.device)
        return color[0], other.clamp_(0.0, 1.0).to(color.dtype)
    return color[0], depth[0], mv[0]


def prepare(case, seed):
    kind, W, H, dev = case["kind"], case["W"], case["H"], _dev()
    st = {"kind": kind, "case": case, "in": _inputs(case, seed)}
    cdt = CDT[case["dtype"]]
    if kind == "frames":
        F = case["frames"]
        st["out"] = torch.empty((F, 3, 3, H, W), dtype=DT[case["dtype"]], device=dev)
        st["mask"] = torch.empty((F, 3, H, W), dtype=torch.uint8, device=dev)
        st["ws"] = binding.workspace(binding.exw_workspace_bytes(binding.OP_EXTRAPOLATE, W, H, cdt, F, 3), dev)
    elif kind == "batched":
        st["bufs"], st["streams"], st["outs"] = [], [], []
        for color, depth, mv in st["in"]:
            n, h, w = depth.shape
            out = torch.empty((n, 3, 3, h, w), dtype=color.dtype, device=dev)
            mask = torch.empty((n, 3, h, w), dtype=torch.uint8, device=dev)
            st["bufs"].append((out, mask))
            for i in range(n):
                st["streams"].append((color[i], depth[i], mv[i]))
                st["outs"].append((out[i], mask[i]))
        st["ws"] = binding.workspace(binding.exw_batched_workspace_bytes(st["streams"], 3), dev)
    elif kind == "train":
        st["ws"] = binding.workspace(binding.exw_workspace_bytes(binding.OP_WARP_L2_GRAD, W, H, cdt, 1, 3), dev)
    elif kind == "autograd":
        st["color"] = st["in"][0].clone().requires_grad_(True)
        st["mv"] = st["in"][2].clone().requires_grad_(True)
    elif kind == "recursive":
        n = case["steps"]
        st["out"] = torch.empty((n, 3, H, W), dtype=DT[case["dtype"]], device=dev)
        st["mask"] = torch.empty((n, H, W), dtype=torch.uint8, device=dev)
        st["ws"] = binding.workspace(binding.exw_workspace_bytes(binding.OP_WARP_RECURSIVE, W, H, cdt), dev)
    elif kind == "staged":
        st["keys"] = torch.empty((H, W), dtype=torch.int64, device=dev)
        st["out"] = torch.empty((3, H, W), dtype=DT[case["dtype"]], device=dev)
        st["mask"] = torch.empty((H, W), dtype=torch.uint8, device=dev)
        st["ws"] = binding.workspace(binding.exw_workspace_bytes(binding.OP_FILL_HOLES, W, H, cdt), dev)
    else:
        st["ws"] = binding.workspace(binding.exw_workspace_bytes(binding.OP_STATS, W, H), dev)
    return st


def run(st):
    kind, case = st["kind"], st["case"]
    if kind == "frames":
        c, d, m = st["in"]
        return binding.exw_extrapolate(c, d, m, 3, case["fill"], st["out"], st["mask"], st["ws"])
    if kind == "batched":
        binding.exw_extrapolate_batched(st["streams"], 3, outs=st["outs"], ws=st["ws"])
        return st["bufs"]
    if kind == "train":
        c, d, m, t = st["in"]
        return binding.exw_warp_l2_grad(c, d, m, t, 3, ws=st["ws"])
    if kind == "autograd":
        _, d, _, grad = st["in"]
        st["color"].grad = st["mv"].grad = None
        out, mask = autograd.warp(st["color"], d, st["mv"], case["k"])
        out.backward(grad)
        return out.detach(), mask, st["color"].grad, st["mv"].grad
    if kind == "recursive":
        c, d, m = st["in"]
        binding.exw_warp_recursive(c, d, m, case["steps"], True, st["out"], st["mask"], st["ws"])
        return st["out"], st["mask"]
    if kind == "staged":
        c, d, m = st["in"]
        keys = binding.exw_splat_motion(d, m, case["k"], 4, st["keys"])
        out, mask = binding.exw_warp(c, d, m, keys, case["k"], 4, st["out"], st["mask"])
        binding.exw_fill_holes(out, mask, st["ws"])
        return keys, out, mask
    if kind == "features":
        return binding.exw_mv_variance(st["in"][0], st["ws"])
    a, b = st["in"]
    return binding.exw_psnr(a, b, st["ws"]), binding.exw_ssim(a, b, st["ws"])


# ---------------------------------------------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------------------------------------------

def _splat(depth, mv, k):
    """Winners of the forward splat by k/4 of the motion: (winner index or -1) [H*W]."""
    H, W = depth.shape
    dev = depth.device
    y, x = torch.meshgrid(torch.arange(H, device=dev), torch.arange(W, device=dev), indexing="ij")
    ok = torch.isfinite(depth) & (depth > 0) & torch.isfinite(mv).all(0)
    m = torch.where(ok, mv.double(), torch.zeros((), dtype=torch.float64, device=dev)) * (k / 4.0)
    tx, ty = x + torch.floor(0.5 + m[0]).long(), y + torch.floor(0.5 + m[1]).long()
    ok &= (tx >= 0) & (tx < W) & (ty >= 0) & (ty < H)
    key = (depth.contiguous().view(torch.int32).long() << 32) | (y * W + x)
    keys = torch.full((H * W,), torch.iinfo(torch.int64).max, dtype=torch.int64, device=dev)
    keys.scatter_reduce_(0, (ty * W + tx)[ok], key[ok], "amin")
    return torch.where(keys == torch.iinfo(torch.int64).max, -1, keys & 0xFFFFFFFF)


def _gather(color, depth, mv, k):
    """The warp by k/4 in 64 bits: a dict with the colour (0 on holes), the hole mask and what the adjoint needs."""
    H, W = depth.shape
    dev = depth.device
    win = _splat(depth, mv, k)
    empty = win < 0
    p = win.clamp(min=0)
    D, col = depth.double().reshape(-1), color.double().reshape(3, -1)
    Dq = torch.where(empty, math.inf, D[p]).view(H, W)
    pad = torch.nn.functional.pad(Dq[None, None], (1, 1, 1, 1), value=math.inf)[0, 0]
    near = sum(((Dq - n) > Dq / 32.0).int()
               for n in (pad[1:-1, :-2], pad[1:-1, 2:], pad[:-2, 1:-1], pad[2:, 1:-1]))
    crack = (~empty.view(H, W)) & (near >= 3)
    hole = empty | crack.reshape(-1)
    q = torch.arange(H * W, device=dev)
    px, py = p % W, p // W
    m = mv.double().reshape(2, -1)[:, p] * (k / 4.0)
    rx, ry = (q % W - px) - m[0], (q // W - py) - m[1]
    sx, sy = torch.sign(rx).long(), torch.sign(ry).long()
    ex, ey = (sx != 0) & (px + sx >= 0) & (px + sx < W), (sy != 0) & (py + sy >= 0) & (py + sy < H)
    Dp = D[p]
    taps, part = [p], [torch.ones_like(hole)]
    for inside, off in ((ex, sx), (ey, sy * W), (ex & ey, sx + sy * W)):
        t = torch.where(inside, p + off, p)
        taps.append(t)
        part.append(inside & ((D[t] - Dp).abs() <= Dp / 32.0))
    wx1, wy1 = rx.abs(), ry.abs()
    wx0, wy0 = 1.0 - wx1, 1.0 - wy1
    w = [a * b * s for (a, b), s in zip(((wx0, wy0), (wx1, wy0), (wx0, wy1), (wx1, wy1)), part)]
    S = w[0] + w[1] + w[2] + w[3]
    out = sum(wt * col[:, t] for wt, t in zip(w, taps)) / S
    out = torch.where(hole, torch.zeros((), dtype=torch.float64, device=dev), out)
    return {"out": out.view(3, H, W), "hole": hole.view(H, W), "win": win, "p": p, "taps": taps, "part": part, "w": w,
            "S": S, "col": col, "sx": sx, "sy": sy, "w1": (wx0, wx1, wy0, wy1), "k": k}


def _fill(color, hole):
    """Pull-push: a hole takes its first valid ancestor of the halving pyramid (0 when there is none)."""
    levels = [(color * ~hole, (~hole).double())]
    while max(levels[-1][0].shape[1:]) > 1:
        c, v = levels[-1]
        c = torch.nn.functional.pad(c, (0, c.shape[2] % 2, 0, c.shape[1] % 2))
        v = torch.nn.functional.pad(v, (0, v.shape[1] % 2, 0, v.shape[0] % 2))
        n = v[0::2, 0::2] + v[0::2, 1::2] + v[1::2, 0::2] + v[1::2, 1::2]
        s = c[:, 0::2, 0::2] + c[:, 0::2, 1::2] + c[:, 1::2, 0::2] + c[:, 1::2, 1::2]
        levels.append((s / n.clamp(min=1.0), (n > 0).double()))
    up, have = levels[-1]
    for c, v in reversed(levels[:-1]):
        H, W = v.shape
        up = up.repeat_interleave(2, 1).repeat_interleave(2, 2)[:, :H, :W]
        up = torch.where(v > 0, c, up)
    return up


def _adjoint(g, grad, grad_color, grad_mv):
    """Adds the gradients of the warp g for the output gradient grad [3][H*W] (64 bits) to grad_color and grad_mv."""
    live = ~g["hole"].reshape(-1)
    p, S, col, w = g["p"][live], g["S"][live], g["col"], [x[live] for x in g["w"]]
    taps, part = [t[live] for t in g["taps"]], [x[live].double() for x in g["part"]]
    up = grad[:, live]
    out = sum(wt * col[:, t] for wt, t in zip(w, taps)) / S
    for wt, t in zip(w, taps):
        for c in range(3):
            grad_color[c].index_add_(0, t, up[c] * wt / S)
    wx0, wx1, wy0, wy1 = (x[live] for x in g["w1"])
    sx, sy = g["sx"][live].double(), g["sy"][live].double()
    # weights' derivatives: the tap on the residual's side grows with it, the other shrinks
    dx = (-sx * wy0, sx * wy0 * part[1], -sx * wy1 * part[2], sx * wy1 * part[3])
    dy = (-sy * wx0, -sy * wx1 * part[1], sy * wx0 * part[2], sy * wx1 * part[3])
    scale = -g["k"] / 4.0
    for axis, d in enumerate((dx, dy)):
        v = sum((up * dt * (col[:, t] - out)).sum(0) for dt, t in zip(d, taps)) / S
        grad_mv[axis].index_add_(0, p, scale * v)


def exact(case, seed):
    kind = case["kind"]
    data = _inputs(case, seed)
    if kind in ("frames", "batched"):
        fill = case.get("fill", True)

        def frames(color, depth, mv):
            out = torch.empty((color.shape[0], 3) + tuple(color.shape[1:]), dtype=torch.float64, device=color.device)
            for f in range(color.shape[0]):
                for k in (1, 2, 3):
                    g = _gather(color[f], depth[f], mv[f], k)
                    out[f, k - 1] = _fill(g["out"], g["hole"]) if fill else g["out"]
            return out

        return (frames(*data), None) if kind == "frames" else [(frames(*grp), None) for grp in data]
    if kind == "train":
        color, depth, mv, target = data
        F, _, H, W = color.shape
        loss = torch.zeros(F, dtype=torch.float64, device=color.device)
        gc = torch.zeros((F, 3, H * W), dtype=torch.float64, device=color.device)
        gm = torch.zeros((F, 2, H * W), dtype=torch.float64, device=color.device)
        for f in range(F):
            for k in (1, 2, 3):
                g = _gather(color[f], depth[f], mv[f], k)
                d = (g["out"] - target[f, k - 1].double()) * ~g["hole"]
                loss[f] += d.square().sum()
                _adjoint(g, 2.0 * d.reshape(3, -1), gc[f], gm[f])
        return loss, gc.view(F, 3, H, W), gm.view(F, 2, H, W)
    if kind == "autograd":
        color, depth, mv, grad = data
        H, W = depth.shape
        g = _gather(color, depth, mv, case["k"])
        gc = torch.zeros((3, H * W), dtype=torch.float64, device=color.device)
        gm = torch.zeros((2, H * W), dtype=torch.float64, device=color.device)
        _adjoint(g, grad.double().reshape(3, -1), gc, gm)
        return g["out"], None, gc.view(3, H, W), gm.view(2, H, W)
    if kind == "recursive":
        color, depth, mv = data
        outs = []
        for _ in range(case["steps"]):
            g = _gather(color, depth, mv, 1)
            outs.append(_fill(g["out"], g["hole"]))
            hole, p = g["hole"], g["p"].view(depth.shape)
            color = outs[-1]
            mv = torch.where(hole, 0.0, mv.reshape(2, -1)[:, p])
            depth = torch.where(hole, math.nan, depth.reshape(-1)[p])
        return torch.stack(outs), None
    if kind == "staged":
        g = _gather(*data, case["k"])
        return None, _fill(g["out"], g["hole"]), None
    if kind == "features":
        m = data[0].double().reshape(2, -1)
        ok = torch.isfinite(m).all(0)
        m = m[:, ok]
        v = (m - m.mean(1, keepdim=True)).square().mean(1)
        return float(ok.sum()), float(v[0]), float(v[1])
    a, b = (t.double() for t in data)
    mse = float((a - b).square().mean())
    t = torch.arange(-5, 6, dtype=torch.float64, device=a.device)
    win = torch.exp(-t * t / 4.5)
    win /= win.sum()

    def mean(v):
        v = sum(float(win[i]) * v[:, :, i:v.shape[2] - 10 + i] for i in range(11))
        return sum(float(win[i]) * v[:, i:v.shape[1] - 10 + i, :] for i in range(11))

    ma, mb = mean(a), mean(b)
    va, vb, cab = mean(a * a) - ma * ma, mean(b * b) - mb * mb, mean(a * b) - ma * mb
    ssim = ((2 * ma * mb + 1e-4) * (2 * cab + 9e-4)) / ((ma * ma + mb * mb + 1e-4) * (va + vb + 9e-4))
    return -10.0 * math.log10(mse), float(ssim.mean())
