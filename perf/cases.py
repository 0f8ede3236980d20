"""Performance cases: the calls a user of the package makes, over the sizes they make them at.

listed() names them, draw(rng) gives more of the same ranges, prepare(case, seed) builds what a
program holds before the call, run(state) is one pass through the package's public entry points,
work(case) the bytes and operations such a pass cannot do without, and exact(case, seed) its
outputs in float64 from plain torch.

The scenes are box-shaped rooms with box-shaped furniture seen by cameras inside them.  Their
supervision maps (z-depth and camera-frame normals) come from an analytic ray cast, and their
planes are samples of the visible surfaces in one of three states of a fit:
  "plain"    random orientation, radii 0.2 m: the start of the throughput benchmark;
  "mono"     surface orientation up to 8 degrees, radii half the nearest-centre distance: the
             monocular-style start;
  "settled"  surface orientation up to 2 degrees, centres within about 1 cm of the surface, radii
             0.05-0.4 m: planes late in a fit.
Fits run with a learning rate of 0, so that a pass leaves its planes where they are and can be
repeated; everything else of the optimisation step, Adam included, runs as in a fit.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch
import torch.nn.functional as F

DEV = "cuda"
ROOM = (8.0, 10.0, 3.0)
M_NEAREST = 30
Z_NEAR, Z_FAR, W_MIN = float(np.float32(0.01)), 100.0, float(np.float32(1e-4))
A_COS, A_L1N, A_DEPTH = 5.0, 5.0, 1.0        # Eq. 14 weights
PS_HARD, PS_GAUSSIAN, PS_SINGLE = 2, 4, 1    # ps_settings.flags
FLAGS = {"": 0, "single": PS_SINGLE, "gauss": PS_GAUSSIAN, "hard": PS_HARD}
PATCH, SLOTS = 64, 8
WEIGHTS = os.path.join("paper_2412_03451_gb300", "weights", "seednet.npz")


def _fit(name, **kw):
    case = {"name": name, "kind": "fit", "scenes": 1, "planes": 3000, "views": 8, "h": 480, "w": 640, "uneven": False,
            "ite": 0, "start": "plain", "flags": "", "tile_w": 8, "tile_h": 8, "mode": "graph"}
    return case | kw


def _render(name, **kw):
    case = {"name": name, "kind": "render", "planes": 2000, "views": 8, "h": 480, "w": 640, "start": "settled",
            "flags": "", "out": "maps", "tile_w": 16, "tile_h": 16}
    return case | kw


def listed():
    return [
        # one eager optimisation step of the tiny room (the first thing a new user runs, and every
        # test): 64 planes, 8 views of 128x96; launches and host calls count most
        _fit("tiny_step", planes=64, h=96, w=128, tile_w=16, tile_h=16, mode="eager"),
        # the paper-scale room at the first iterations of a fit (blurred weights, long lists),
        # replayed from a CUDA graph as every fit does
        _fit("room_step_first"),
        # the same near the end of a fit (lambda = 300): short lists, most pairs opaque
        _fit("room_step_late", ite=4000, start="settled"),
        # 16 rooms of uneven plane counts and image sizes in one step, a third into the schedule
        _fit("rooms_step", scenes=16, uneven=True, ite=1000, start="settled"),
        # the Gaussian weight of the ablation (Eq. 5) with planes well into a fit, when each of them
        # reaches 4.3 of its radii
        _fit("gauss_step", planes=2000, ite=1000, start="settled", flags="gauss", tile_w=16, tile_h=16),
        # a large scene (10,000 planes, 64 views) through the separate forward, loss and backward
        # kernels, as a program with a loss of its own between them runs it
        _fit("stress_step", planes=10000, views=64, ite=1000, start="settled", mode="separate"),
        # the autograd function: a render and its backward for an arbitrary upstream gradient, at
        # an odd image size
        {"name": "autograd", "kind": "autograd", "planes": 1500, "views": 5, "h": 383, "w": 511, "ite": 500,
         "start": "mono", "tile_w": 16, "tile_h": 16},
        # evaluation: depth and normals of the fitted planes at the sharpest weight, odd sizes
        _render("render_fitted", planes=3000, h=471, w=627),
        # supervision: hard-edged depth and normal maps of every view of a room
        _render("render_hard", views=64, flags="hard"),
        # seed network: every 64x64 patch of a room's 64 views at 640x480
        {"name": "seeds_infer", "kind": "seeds", "patches": 4480, "train": False},
        # one training step of the seed network at its batch size
        {"name": "seeds_train", "kind": "seeds", "patches": 256, "train": True},
        # initial radii of a scene's planes from their nearest centres
        {"name": "start_radii", "kind": "radii", "planes": 3000},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fit", "fit", "fit", "gauss", "separate", "autograd", "render", "render", "infer", "train", "radii"])
    tile_w, tile_h = rng.choice([(8, 8), (8, 8), (16, 16), (16, 16), (32, 8)])
    tile = {"tile_w": tile_w, "tile_h": tile_h}
    w = rng.randint(96, 640)
    size = {"w": w, "h": max(72, w * 3 // 4 - rng.randint(0, 5))}
    start, ite = rng.choice([("plain", rng.randint(0, 400)), ("mono", rng.randint(0, 1500)), ("settled", rng.randint(500, 5000))])
    if kind == "fit":
        scenes = rng.choice([1, 1, 2, 5, 11])
        case = _fit("", scenes=scenes, uneven=scenes > 1, planes=_log_int(rng, 64, 5000 if scenes == 1 else 3000), ite=ite, start=start,
                    views=_log_int(rng, 2, 16 if scenes == 1 else 8), flags=rng.choice(["", "", "", "single"]),
                    mode=rng.choice(["graph", "graph", "eager"]), **size, **tile)
    elif kind == "gauss":
        case = _fit("", planes=_log_int(rng, 64, 2000), views=_log_int(rng, 2, 8), ite=ite, flags="gauss", start=start, **size, **tile)
    elif kind == "separate":
        case = _fit("", planes=_log_int(rng, 500, 10000), views=_log_int(rng, 4, 48), ite=ite, start=start, mode="separate", **size, **tile)
    elif kind == "autograd":
        case = {"kind": kind, "planes": _log_int(rng, 64, 3000), "views": _log_int(rng, 1, 16), "ite": ite, "start": start, **size, **tile}
    elif kind == "render":
        case = _render("", planes=_log_int(rng, 64, 5000), views=_log_int(rng, 1, 64), flags=rng.choice(["", "hard"]),
                       out=rng.choice(["maps", "ids"]), **size, **tile)
    elif kind == "infer":
        case = {"kind": "seeds", "patches": 64 * _log_int(rng, 1, 70), "train": False}
    elif kind == "train":
        case = {"kind": "seeds", "patches": 64 * rng.randint(1, 4), "train": True}
    else:
        case = {"kind": kind, "planes": _log_int(rng, 200, 20000)}
    case.pop("name", None)
    return case


# ---------------------------------------------------------------------------
# Scenes.

def _shapes(case):
    """Per scene (planes, h, w): an uneven batch mixes plane counts and three image sizes."""
    n = case.get("scenes", 1)
    if not case.get("uneven"):
        return [(case["planes"], case["h"], case["w"])] * n
    return [(max(16, case["planes"] * (s + 1) // n), case["h"] * (2 + s % 3) // 4, case["w"] * (2 + s % 3) // 4) for s in range(n)]


def _boxes(rng):
    """[n, 2, 3] corners of the furniture, all lower than the cameras."""
    n = int(rng.integers(6, 11))
    size = rng.uniform([0.4, 0.4, 0.3], [2.0, 2.0, 1.1], size=(n, 3))
    lo = rng.uniform(0.05, 1.0, size=(n, 3)) * (np.asarray(ROOM) - size - 0.05)
    lo[:, 2] = 0.0
    return np.stack([lo, lo + size], 1)


def _cameras(rng, views, h, w):
    """World-to-camera [views, 3, 4] and intrinsics [views, 4] (x right, y down, z forward)."""
    eye = rng.uniform([1.0, 1.0, 1.3], [ROOM[0] - 1.0, ROOM[1] - 1.0, 1.8], size=(views, 3))
    yaw, pitch = rng.uniform(0, 2 * np.pi, views), np.deg2rad(rng.uniform(-25, 5, views))
    fwd = np.stack([np.cos(yaw) * np.cos(pitch), np.sin(yaw) * np.cos(pitch), np.sin(pitch)], 1)
    right = np.cross(fwd, [0.0, 0.0, 1.0])
    right /= np.linalg.norm(right, axis=1, keepdims=True)
    R = np.stack([right, np.cross(fwd, right), fwd], 1)
    w2c = np.concatenate([R, -np.einsum("vij,vj->vi", R, eye)[:, :, None]], 2)
    f = 500.0 * w / 640.0
    return w2c.astype(np.float32), np.tile(np.array([f, f, w / 2.0, h / 2.0], np.float32), (views, 1))


def _rays(intr, h, w):
    """Ray directions [h, w, 3] through the pixel centres of one view, z = 1, float64."""
    fx, fy, cx, cy = (float(v) for v in intr)
    x = (torch.arange(w, device=DEV, dtype=torch.float64) + 0.5 - cx) / fx
    y = (torch.arange(h, device=DEV, dtype=torch.float64) + 0.5 - cy) / fy
    return torch.stack([x.expand(h, w), y[:, None].expand(h, w), torch.ones(h, w, device=DEV, dtype=torch.float64)], -1)


def _cast(boxes, w2c, intr, h, w):
    """Supervision of all views: z-depth [V*h*w] and camera-frame normals [V*h*w, 3], float32."""
    depth, normal = [], []
    lo = torch.tensor(np.concatenate([np.zeros((1, 3)), boxes[:, 0]]), device=DEV)
    hi = torch.tensor(np.concatenate([[ROOM], boxes[:, 1]]), device=DEV)
    for T, K in zip(w2c.astype(np.float64), intr):
        R = torch.tensor(T[:, :3], device=DEV)
        eye = torch.tensor(-T[:, :3].T @ T[:, 3], device=DEV)
        d = (_rays(K, h, w).reshape(-1, 3) @ R)[:, None]                     # world directions
        a, b = (lo - eye) / d, (hi - eye) / d
        near, far = torch.minimum(a, b), torch.maximum(a, b)
        tin, ain = near.max(-1)
        tout, aout = far.min(-1)
        t = torch.where((tin > 0) & (tin < tout), tin, torch.full_like(tin, math.inf))
        t[:, 0], axis = tout[:, 0], ain
        axis[:, 0] = aout[:, 0]                                              # the room is seen from inside
        t, k = t.min(-1)
        axis = axis.gather(1, k[:, None])
        n = torch.zeros_like(d[:, 0]).scatter_(1, axis, -torch.sign(d[:, 0].gather(1, axis)))
        depth.append(t.float())
        normal.append((n @ R.T).float())
    return torch.cat(depth), torch.cat(normal)


def _quat(R):
    """Unit quaternions (w, x, y, z) of rotations [n, 3, 3] that are not half turns about an axis
    of the frame: the largest of the four candidate vectors."""
    m = R.reshape(-1, 9).T
    q = np.stack([
        np.stack([1 + m[0] + m[4] + m[8], m[7] - m[5], m[2] - m[6], m[3] - m[1]], 1),
        np.stack([m[7] - m[5], 1 + m[0] - m[4] - m[8], m[1] + m[3], m[2] + m[6]], 1),
        np.stack([m[2] - m[6], m[1] + m[3], 1 - m[0] + m[4] - m[8], m[5] + m[7]], 1),
        np.stack([m[3] - m[1], m[2] + m[6], m[5] + m[7], 1 - m[0] - m[4] + m[8]], 1)], 1)
    norm = np.linalg.norm(q, axis=2)
    best = norm.argmax(1)
    return q[np.arange(len(q)), best] / norm.max(1)[:, None]


def _planes(rng, boxes, n, start):
    """Centres [n, 3], quaternions [n, 4] and radii [n, 4] of planes on the room's surfaces."""
    lo = np.concatenate([np.zeros((1, 3)), boxes[:, 0]])
    hi = np.concatenate([[ROOM], boxes[:, 1]])
    face = np.array([(b, ax, s) for b in range(len(lo)) for ax in range(3) for s in (0, 1) if b == 0 or (ax, s) != (2, 0)])
    ext = (hi - lo)[face[:, 0]]
    area = ext.prod(1) / ext[np.arange(len(face)), face[:, 1]]
    pick = face[rng.choice(len(face), size=n, p=area / area.sum())]
    b, ax, s = pick.T
    c = lo[b] + rng.uniform(size=(n, 3)) * (hi - lo)[b]
    c[np.arange(n), ax] = np.where(s == 0, lo[b, ax], hi[b, ax])
    nrm = np.zeros((n, 3))
    nrm[np.arange(n), ax] = np.where((s == 0) == (b == 0), 1.0, -1.0)        # towards the free space
    if start == "plain":
        q = rng.normal(size=(n, 4))
        radii = np.full((n, 4), 0.2)
    else:
        tilt, off = (np.deg2rad(8.0), 0.05) if start == "mono" else (np.deg2rad(2.0), 0.01)
        nrm = nrm + rng.normal(size=(n, 3)) * tilt / math.sqrt(2.0)
        nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
        vx = np.cross(nrm, rng.normal(size=(n, 3)))
        vx /= np.linalg.norm(vx, axis=1, keepdims=True)
        q = _quat(np.stack([vx, np.cross(nrm, vx), nrm], 2))
        c = c + nrm * rng.normal(size=(n, 1)) * off
        if start == "mono":
            p = torch.tensor(c, device=DEV)
            near = torch.cat([torch.cdist(x, p).kthvalue(min(2, n), 1).values for x in p.split(1024)])
            radii = np.repeat((0.5 * near).clamp(0.02, 2.0).cpu().numpy()[:, None], 4, 1)
        else:
            radii = rng.uniform(0.05, 0.4, size=(n, 4))
    return [x.astype(np.float32) for x in (c, q, radii)]


def _scene(case, seed):
    """All scenes of a case: planes, cameras and supervision, as float32 arrays."""
    rng = np.random.default_rng([seed, 7])
    s = {"c": [], "q": [], "r": [], "w2c": [], "intr": [], "H": [], "W": [], "sov": [], "gd": [], "gn": [], "K": []}
    for i, (K, h, w) in enumerate(_shapes(case)):
        boxes = _boxes(rng)
        w2c, intr = _cameras(rng, case["views"], h, w)
        for key, v in zip("cqr", _planes(rng, boxes, K, case["start"])):
            s[key].append(v)
        if case["kind"] == "fit":
            gd, gn = _cast(boxes, w2c, intr, h, w)
            s["gd"].append(gd)
            s["gn"].append(gn)
        s["K"].append(K)
        s["w2c"].append(w2c)
        s["intr"].append(intr)
        s["H"] += [h] * case["views"]
        s["W"] += [w] * case["views"]
        s["sov"] += [i] * case["views"]
    for key in ("c", "q", "r", "w2c", "intr"):
        s[key] = np.concatenate(s[key])
    for key in ("gd", "gn"):
        s[key] = torch.cat(s[key]) if s[key] else None
    return s


def _lam(ite):
    return min(20.0 * math.exp(-(1.0 - 0.001 * ite)), 300.0)                 # Eq. 10


def _upstream(case, seed):
    """An arbitrary gradient of (depth, normal) for the autograd case."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    n = case["views"] * case["h"] * case["w"]
    return torch.randn(n, device=DEV, generator=g), torch.randn(n, 3, device=DEV, generator=g)


def _patches(case, seed):
    """Seed-network inputs [n, 64, 64, 4] bf16 (depth over its median minus 1, normals) cut from
    supervision maps, and training targets [n, 8, 12]."""
    rng = np.random.default_rng([seed, 11])
    n = case["patches"]
    views = -(-n // 70)
    w2c, intr = _cameras(rng, views, 448, 640)
    d, m = _cast(_boxes(rng), w2c, intr, 448, 640)
    d = d.view(views, 7, 64, 10, 64).transpose(2, 3).reshape(-1, 64, 64)[:n]
    m = m.view(views, 7, 64, 10, 64, 3).transpose(2, 3).reshape(-1, 64, 64, 3)[:n]
    ref = d.flatten(1).median(1).values[:, None, None]
    x = torch.cat([(d / ref - 1.0)[..., None], m], -1).bfloat16().contiguous()
    t = np.zeros((n, SLOTS, 12), np.float32)
    t[..., 0] = np.arange(SLOTS) < rng.integers(1, SLOTS + 1, size=(n, 1))   # the largest segments come first
    t[..., 1:4] = rng.normal(size=(n, SLOTS, 3)) * [0.5, 0.5, 0.1]
    q = rng.normal(size=(n, SLOTS, 4))
    t[..., 4:8] = q / np.linalg.norm(q, axis=-1, keepdims=True)
    t[..., 8:12] = rng.normal(-2.0, 0.7, size=(n, SLOTS, 4))
    return x, torch.from_numpy(t).to(DEV)


def _centres(case, seed):
    rng = np.random.default_rng([seed, 13])
    return torch.from_numpy(_planes(rng, _boxes(rng), case["planes"], "settled")[0]).to(DEV)


# ---------------------------------------------------------------------------
# The calls.

def prepare(case, seed):
    from paper_2412_03451_gb300 import seed_train, splat
    kind = case["kind"]
    if kind == "radii":
        return {"kind": kind, "centres": _centres(case, seed)}
    if kind == "seeds":
        net = seed_train.load()
        x, t = _patches(case, seed)
        if not case["train"]:
            net.forward(x)                       # the network's buffers for this batch
        return {"kind": kind, "net": net, "x": x, "t": t, "train": case["train"]}
    s = _scene(case, seed)
    r = splat.Renderer(s["H"], s["W"], s["sov"], np.concatenate([[0], np.cumsum(s["K"])]),
                       tile=(case["tile_w"], case["tile_h"]), flags=FLAGS[case.get("flags", "")])
    flat = splat.planes_to_flat(s["c"], s["q"], s["r"], DEV)
    lam = 300.0 if kind == "render" else _lam(case["ite"])
    if kind == "fit" and case["mode"] == "graph":
        r.preplan([s["w2c"]], [s["intr"]])
    else:
        r.set_cameras(s["w2c"], s["intr"])
    r.ensure_capacity(flat, lam)
    state = {"kind": kind, "r": r, "flat": flat, "lam": lam}
    if kind == "fit":
        fit = splat.Fitter(r, flat, lr=0.0, fused=case["mode"] != "separate")
        fit.lam_offset = case["ite"]
        if case["mode"] == "graph":
            fit.enable_graphs(1, [0], [(s["gd"], s["gn"])])
        state |= {"fit": fit, "gd": s["gd"], "gn": s["gn"], "mode": case["mode"]}
    elif kind == "autograd":
        state |= {"flat": flat.requires_grad_(True), "up": _upstream(case, seed)}
    else:
        state |= {"ids": case["out"] == "ids", "hard": case["flags"] == "hard"}
    return state


def run(state):
    from paper_2412_03451_gb300 import splat, starts
    kind = state["kind"]
    if kind == "radii":
        return starts.nn_radii(state["centres"])
    if kind == "seeds":
        net = state["net"]
        out = net.forward(state["x"])
        if not state["train"]:
            return out
        net.grad.zero_()
        sums = net.loss_backward(state["t"])
        net.adam(lr=0.0)
        return {"out": out, "grad": net.grad, "sums": sums, "m": net.m, "v": net.v}
    r, flat, lam = state["r"], state["flat"], state["lam"]
    if kind == "fit":
        fit = state["fit"]
        if state["mode"] == "graph":
            sums = fit.replay(0)
        else:
            sums = fit.step(state["gd"], state["gn"], lam=lam)
        out = {"grad": fit.grad, "m": fit.m, "v": fit.v, "sums": sums.float()}
        return out | ({"depth": r.depth, "normal": r.normal} if state["mode"] == "separate" else {})
    if kind == "autograd":
        depth, normal = splat.PlaneSplatFunction.apply(flat, r, lam)
        (grad,) = torch.autograd.grad([depth, normal], [flat], state["up"])
        return {"depth": depth.detach(), "normal": normal.detach(), "grad": grad}
    if state["ids"]:
        ids, depth = r.plane_ids(flat, lam, hard=state["hard"])
        return {"ids": ids, "depth": depth}
    depth, normal = r.forward(flat, lam, alpha=False)
    return {"depth": depth, "normal": normal}


def work(case):
    """Each input read once and each output written once; for a render, one evaluated and one
    composited plane per pixel (the paper's formulas: 27 operations to evaluate a pair, 12 to
    composite it, 66 for its gradient), the least that a covered pixel needs."""
    kind = case["kind"]
    if kind == "radii":
        return {"bytes": 28 * case["planes"], "flops": 8 * case["planes"]}
    if kind == "seeds":
        n = case["patches"]
        conv = 2 * 64 * (36 * 1024 + 576 * (256 + 64 + 16)) + 2 * 64 * 96    # operations per patch
        params = 64 * 36 + 3 * 64 * 576 + 64 * 96 + 4 * 64 + 96
        first = 2 * 64 * 36 * 1024                                           # no gradient of the input is needed
        if not case["train"]:
            return {"bytes": 2 * 64 * 64 * 4 * n + 4 * 96 * n + 4 * params, "flops": conv * n}
        return {"bytes": (2 * 64 * 64 * 4 + 4 * 96 * 3) * n + 4 * 7 * params, "flops": (3 * conv - first) * n}
    pix = sum(h * w for _, h, w in _shapes(case)) * case["views"]
    P = sum(k for k, _, _ in _shapes(case))
    if kind == "fit":
        maps = 16 if case["mode"] == "separate" else 0
        return {"bytes": (16 + maps) * pix + 7 * 44 * P, "flops": 105 * pix}
    if kind == "autograd":
        return {"bytes": 32 * pix + 88 * P, "flops": 105 * pix}
    return {"bytes": (8 if case["out"] == "ids" else 16) * pix + 44 * P, "flops": 39 * pix}


# ---------------------------------------------------------------------------
# The same in float64.

def _axes(q):
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    vx = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y + w * z), 2 * (x * z - w * y)], 1)
    vy = torch.stack([2 * (x * y - w * z), 1 - 2 * (x * x + z * z), 2 * (y * z + w * x)], 1)
    return vx, vy, torch.stack([2 * (x * z + w * y), 2 * (y * z - w * x), 1 - 2 * (x * x + y * y)], 1)


def _record(c, q, r, T, single):
    """Planes in the camera frame: centre, v^x, v^y, n, radii."""
    R, t = T[:, :3], T[:, 3]
    vx, vy, n = (a @ R.T for a in _axes(q))
    if single:
        r = r[:, [0, 0, 2, 2]]
    return c @ R.T + t, vx, vy, n, r


def _pair(d, rec, lam, flags):
    """Depth and weight (0 where the filter drops the pair) of rays d against planes, broadcast."""
    p, vx, vy, n, r = rec
    den = (d * n).sum(-1)
    t = (n * p).sum(-1) / den
    o = t[..., None] * d - p
    X, Y = (o * vx).sum(-1), (o * vy).sum(-1)
    sx, sy = torch.where(X > 0, r[..., 0], r[..., 1]), torch.where(Y > 0, r[..., 2], r[..., 3])
    if flags == "gauss":
        w = torch.exp(-0.5 * ((X / sx) ** 2 + (Y / sy) ** 2))
    else:
        m = torch.minimum(sx - X.abs(), sy - Y.abs())
        w = torch.where(m >= 0, torch.ones_like(m), torch.zeros_like(m) if flags == "hard" else 2 * torch.sigmoid(5 * lam * m))
    ok = (den.abs() > 1e-6) & (t > Z_NEAR) & (t < Z_FAR) & (w >= W_MIN)
    return t, torch.where(ok, w, torch.zeros_like(w)), ok


def _in_band(rec, d, reach):
    """Planes whose bounding sphere meets the pyramid of the rays d [h, w, 3]."""
    p = rec[0]
    keep = p[:, 2] > -reach
    for ax in (0, 1):
        lo, hi = float(d[..., ax].min()), float(d[..., ax].max())
        keep &= (p[:, ax] - lo * p[:, 2]) / math.hypot(1, lo) >= -reach
        keep &= (p[:, ax] - hi * p[:, 2]) / math.hypot(1, hi) <= reach
    return keep.nonzero()[:, 0]


def _exact_views(case, s, lam, upstream):
    """Depth and normal maps of every view, the gradient of the flat parameter buffer and the
    per-view loss sums.  upstream(view, rows, D, N) gives (dL/dD, dL/dN, sums) or None."""
    flags = case.get("flags", "")
    c, q, r = (torch.tensor(s[k], device=DEV, dtype=torch.float64, requires_grad=upstream is not None) for k in "cqr")
    grads = [torch.zeros_like(x) for x in (c, q, r)]
    first = np.concatenate([[0], np.cumsum(s["K"])])
    depth, normal, sums = [], [], []
    for v, sc in enumerate(s["sov"]):
        h, w = s["H"][v], s["W"][v]
        rays = _rays(s["intr"][v], h, w)
        T = torch.tensor(s["w2c"][v], device=DEV, dtype=torch.float64)
        ids = torch.arange(first[sc], first[sc + 1], device=DEV)
        total = torch.zeros(4, device=DEV, dtype=torch.float64)
        with torch.no_grad():
            rec = _record(c[ids], q[ids], r[ids], T, flags == "single")
            reach = rec[4].reshape(-1, 2, 2).max(2).values.norm(dim=1)
            reach = reach * math.sqrt(2 * math.log(1 / W_MIN)) * 1.001 if flags == "gauss" else reach + 1.5 * 10.0 / (5 * lam)
        step = max(1, 8192 // w)
        for y in range(0, h, step):
            d = rays[y:y + step]
            near = ids[_in_band(rec, d, reach)]
            d = d.reshape(-1, 1, 3)
            rows = slice(y * w, y * w + len(d))
            if not len(near):
                depth.append(torch.zeros(len(d), device=DEV, dtype=torch.float64))
                normal.append(torch.zeros(len(d), 3, device=DEV, dtype=torch.float64))
                if upstream is not None:
                    total += upstream(v, rows, depth[-1], normal[-1])[2]
                continue
            with torch.no_grad():
                t, _, ok = _pair(d, _record(c[near], q[near], r[near], T, flags == "single"), lam, flags)
                t = torch.where(ok, t, torch.full_like(t, math.inf))
                pick = t.topk(min(M_NEAREST, len(near)), 1, largest=False).indices
                del t, ok
            with torch.set_grad_enabled(upstream is not None):
                rn = _record(c[near], q[near], r[near], T, flags == "single")
                t, wt, ok = _pair(d, [x[pick] for x in rn], lam, flags)
                t = torch.where(ok, t, torch.zeros_like(t))
                tr = torch.cumprod(torch.cat([torch.ones_like(wt[:, :1]), 1 - wt[:, :-1]], 1), 1)
                D = (tr * wt * t).sum(1)
                N = ((tr * wt)[..., None] * rn[3][pick]).sum(1)
                if upstream is not None:
                    gD, gN, part = upstream(v, rows, D.detach(), N.detach())
                    total += part
                    for acc, g in zip(grads, torch.autograd.grad([D, N], [c, q, r], [gD, gN])):
                        acc += g
            depth.append(D.detach())
            normal.append(N.detach())
        sums.append(total)
    grad = torch.cat([g.reshape(-1) for g in grads])
    return torch.cat(depth), torch.cat(normal), grad, torch.stack(sums)


def _exact_fit(case, s):
    off = np.concatenate([[0], np.cumsum([h * w for h, w in zip(s["H"], s["W"])])])

    def eq14(v, rows, D, N):
        at = slice(off[v] + rows.start, off[v] + rows.stop)
        gd, gn = s["gd"][at].double(), s["gn"][at].double()
        ok = (gd > 0).double()
        cos, e, dd = 1 - (N * gn).sum(1), N - gn, D - gd
        gN = -A_COS * torch.sign(cos)[:, None] * gn + A_L1N * torch.sign(e)
        part = torch.stack([(ok * cos.abs()).sum(), (ok * e.abs().sum(1)).sum(), (ok * dd.abs()).sum(), ok.sum()])
        return ok * A_DEPTH * torch.sign(dd), ok[:, None] * gN, part

    lam = float(np.float32(_lam(case["ite"])))
    depth, normal, grad, sums = _exact_views(case, s, lam, eq14)
    out = {"grad": grad, "m": 0.1 * grad, "v": 0.001 * grad * grad, "sums": sums}
    return out | ({"depth": depth, "normal": normal} if case["mode"] == "separate" else {})


def _exact_seeds(case, seed):
    x, tgt = _patches(case, seed)
    p = torch.tensor(np.load(WEIGHTS)["params"], device=DEV, dtype=torch.float64, requires_grad=case["train"])
    y, at = x.double().permute(0, 3, 1, 2), 0

    def take(*shape):
        nonlocal at
        at += math.prod(shape)
        return p[at - math.prod(shape):at].view(*shape)

    def net(y):
        for cin in (4, 64, 64, 64):
            W, b = take(64, 9, cin), take(64)
            cols = F.unfold(y, 3, padding=1, stride=2).view(len(y), cin, 9, -1).transpose(1, 2).reshape(len(y), 9 * cin, -1)
            side = y.shape[-1] // 2
            y = torch.relu(W.reshape(64, -1) @ cols + b[:, None]).view(len(y), 64, side, side)
        W, b = take(96, 64), take(96)
        return y.mean((2, 3)) @ W.T + b

    if not case["train"]:
        with torch.no_grad():
            outs = []
            for part in y.split(256):
                at = 0
                outs.append(net(part))
            return torch.cat(outs)
    out = net(y)
    o, t = out.view(-1, SLOTS, 12), tgt.double()
    valid = t[..., 0]
    bce = F.binary_cross_entropy_with_logits(o[..., 11], valid, reduction="sum")
    q = o[..., 3:7] / o[..., 3:7].norm(dim=-1, keepdim=True)
    on = (valid > 0.5).double()
    terms = torch.stack([bce, (on * (o[..., :3] - t[..., 1:4]).abs().sum(-1)).sum(),
                         (on * (1 - (q * t[..., 4:8]).sum(-1).abs())).sum(),
                         (on * 0.5 * (o[..., 7:11] - t[..., 8:12]).abs().sum(-1)).sum()])
    (grad,) = torch.autograd.grad(terms.sum() / len(out), p)
    return {"out": out.detach(), "grad": grad, "sums": terms.detach(), "m": 0.1 * grad, "v": 0.001 * grad * grad}


def exact(case, seed):
    kind = case["kind"]
    if kind == "radii":
        p = _centres(case, seed).double()
        near = torch.cat([torch.cdist(x, p, compute_mode="donot_use_mm_for_euclid_dist").kthvalue(2, 1).values for x in p.split(512)])
        return (0.5 * near).clamp(0.02, 2.0)[:, None].expand(-1, 4).contiguous()
    if kind == "seeds":
        return _exact_seeds(case, seed)
    s = _scene(case, seed)
    if kind == "fit":
        return _exact_fit(case, s)
    if kind == "render":
        depth, normal, _, _ = _exact_views(case, s, 300.0, None)
        return {"ids": None, "depth": depth} if case["out"] == "ids" else {"depth": depth, "normal": normal}
    gD, gN = (g.double() for g in _upstream(case, seed))
    n = case["h"] * case["w"]

    def given(v, rows, D, N):
        at = slice(v * n + rows.start, v * n + rows.stop)
        return gD[at], gN[at], torch.zeros(4, device=DEV, dtype=torch.float64)

    depth, normal, grad, _ = _exact_views(case, s, float(np.float32(_lam(case["ite"]))), given)
    return {"depth": depth, "normal": normal, "grad": grad}
