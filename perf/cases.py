"""Performance cases of the rasterizer and the mapping / refinement path around it.

A case is one pass of what a program built on this package does over and over: render keyframes and
back-propagate a mapping loss to the Gaussians and the camera poses, render views alone, evaluate a
loss, step the optimiser, form the pose graph's photometric blocks, fuse two submaps.  Scenes are
drawn on the GPU from the seed alone, shaped like the package's synthetic workloads: a cloud in
front of a camera, box rooms with furniture, several agents' rooms of uneven size, a floor of rooms.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch
import torch.nn.functional as F

from paper_2605_10760_gb300 import raster as R
from paper_2605_10760_gb300 import scenes as S

FIELDS = ("means", "log_scales", "quats", "opacities", "colors")
AGENTS = (50_000, 80_000, 120_000, 160_000, 200_000, 260_000, 330_000, 400_000)


# ------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------

def _frame(name, scene, n, views, w, h, **over):
    return {"name": name, "kind": "frame", "scene": scene, "n": n, "views": views, "w": w, "h": h, "loss": "l1_fused",
            "depth_w": 0.1, "tile_w": 16, "tile_h": 16, "bg": 0.0, "call": "eager", **over}


def listed():
    return [
        # the smallest differentiable render: a couple of thousand Gaussians through torch.autograd, as
        # an interactive fit or a test of a new term calls it (host work and launches count)
        _frame("autograd_cloud2k", "cloud", 2_000, 1, 320, 240, loss="upstream", call="autograd"),
        # the plain single-view rasterizer: 10k Gaussians, few tiles with long lists, L1 on RGB
        _frame("step_cloud10k", "cloud", 10_000, 1, 320, 240, loss="l1", depth_w=0.0),
        # the headline: one keyframe of a Replica-shaped room, RGB + depth L1, pose gradient, the
        # whole step replayed as one CUDA graph
        _frame("step_room500k", "room", 500_000, 1, 1200, 680, call="graph"),
        # odd image size, two views, all three upstream gradients, a background and the wide tile,
        # through torch.autograd with its capacity check
        _frame("autograd_room120k_odd", "room", 120_001, 2, 641, 479, loss="upstream", call="autograd", bg=0.4,
               tile_w=32, depth_w=0.3),
        # rendering alone: four frames of a trajectory through a submap (evaluation, keyframe depth maps)
        _frame("render_room260k", "room", 260_000, 4, 1200, 680, loss="none"),
        # one batched mapping step of eight agents, four keyframes each, submaps of uneven size
        _frame("step_agents8x4", "agents", sum(AGENTS), 32, 1200, 680),
        # the mapping loop's render, L1 + SSIM loss and backward over a window of eight keyframes
        _frame("map_room1m", "room", 1_000_000, 8, 1200, 680, loss="ssim", depth_w=0.0),
        # the fused global map: every agent's keyframes in one launch, pose gradients of all of them
        _frame("step_floor4m", "floor", 4_000_000, 64, 1200, 680),
        # the optimiser step of the mapping loop with the isotropy regulariser
        {"name": "adam_room1m", "kind": "adam", "n": 1_000_000, "iso": 10.0},
        # the refinement loss on eight exposure-compensated keyframes, then the normal term
        {"name": "refine_loss_8views", "kind": "loss", "views": 8, "w": 1200, "h": 680, "normal": True},
        # the pose graph's photometric blocks: eight anchor pairs, both directions
        {"name": "pho_16edges", "kind": "pho", "edges": 16, "w": 1200, "h": 680, "stride": 1},
        # occupancy-aware fusion of two aligned submaps with eight keyframe depth maps
        {"name": "fuse_2m", "kind": "fuse", "n": 2_000_000, "views": 8, "w": 1200, "h": 680, "stride": 2},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(("frame",) * 6 + ("adam", "loss", "pho", "fuse"))
    w, h = _log(rng, 160, 1200), _log(rng, 120, 680)
    if kind == "adam":
        return {"kind": kind, "n": _log(rng, 1_000, 2_000_000), "iso": rng.choice((0.0, 10.0))}
    if kind == "loss":
        return {"kind": kind, "views": rng.randint(1, 8), "w": w, "h": h, "normal": rng.random() < 0.5}
    if kind == "pho":
        return {"kind": kind, "edges": rng.randint(1, 16), "w": w, "h": h, "stride": rng.choice((1, 1, 2, 3))}
    if kind == "fuse":
        return {"kind": kind, "n": _log(rng, 10_000, 2_000_000), "views": rng.randint(1, 8), "w": w, "h": h,
                "stride": rng.choice((1, 2, 4))}
    scene = rng.choice(("cloud", "room", "room", "agents", "floor"))
    n = {"cloud": (500, 40_000), "room": (20_000, 1_000_000), "agents": (100_000, 1_600_000),
         "floor": (200_000, 2_000_000)}[scene]
    views = {"cloud": rng.choice((1, 1, 2)), "room": _log(rng, 1, 8), "agents": 8 * rng.randint(1, 4),
             "floor": _log(rng, 4, 32)}[scene]
    tile = rng.choice(((16, 16), (16, 16), (16, 16), (16, 8), (32, 16)))
    loss, call = rng.choice((("l1_fused", "eager"), ("l1_fused", "graph"), ("l1", "eager"), ("ssim", "eager"),
                             ("none", "eager"), ("upstream", "autograd")))
    return {"kind": kind, "scene": scene, "n": _log(rng, *n), "views": views, "w": w, "h": h, "loss": loss, "call": call,
            "depth_w": rng.choice((0.0, 0.1)), "tile_w": tile[0], "tile_h": tile[1], "bg": rng.choice((0.0, 0.0, 0.4))}


# ------------------------------------------------------------------------------------------
# seeded inputs
# ------------------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * int(seed) + 17)
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda")


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _wave(g, pts, lo, hi, scale):
    """Smooth values of points [..., D]: a few random plane waves per channel, mapped into [lo, hi]."""
    k = scale * _randn(g, pts.shape[-1], 6)
    ph = 6.2832 * _rand(g, 6)
    return lo + (hi - lo) * (0.5 + 0.5 * torch.sin(pts @ k + ph).mean(-1))


def _room(rng, x0, y0, size, n_boxes):
    """Faces (origin, edge, edge, normal) of a box room and its furniture, as [F, 4, 3]."""
    lx, ly, lz = size
    out = []
    for z, s in ((0.0, 1.0), (lz, -1.0)):
        out.append(((x0, y0, z), (lx, 0, 0), (0, ly, 0), (0, 0, s)))
    for x, s in ((x0, 1.0), (x0 + lx, -1.0)):
        out.append(((x, y0, 0), (0, ly, 0), (0, 0, lz), (s, 0, 0)))
    for y, s in ((y0, 1.0), (y0 + ly, -1.0)):
        out.append(((x0, y, 0), (lx, 0, 0), (0, 0, lz), (0, s, 0)))
    for _ in range(n_boxes):
        a, b, c = rng.uniform(0.3, 1.5), rng.uniform(0.3, 1.5), rng.uniform(0.3, 1.2)
        bx, by = x0 + rng.uniform(0, lx - a), y0 + rng.uniform(0, ly - b)
        out += [((bx, by, c), (a, 0, 0), (0, b, 0), (0, 0, 1)),
                ((bx, by, 0), (0, b, 0), (0, 0, c), (-1, 0, 0)), ((bx + a, by, 0), (0, b, 0), (0, 0, c), (1, 0, 0)),
                ((bx, by, 0), (a, 0, 0), (0, 0, c), (0, -1, 0)), ((bx, by + b, 0), (a, 0, 0), (0, 0, c), (0, 1, 0))]
    return out


def _matrix_to_quat(M):
    """Quaternions (w, x, y, z) of rotation matrices [N, 3, 3]: the largest of the four squared terms leads."""
    d = torch.stack([M[:, 0, 0], M[:, 1, 1], M[:, 2, 2]], 1)
    tr = d.sum(1)
    sq = torch.stack([1 + tr, 1 + 2 * d[:, 0] - tr, 1 + 2 * d[:, 1] - tr, 1 + 2 * d[:, 2] - tr], 1)
    a, b, c = M[:, 2, 1] - M[:, 1, 2], M[:, 0, 2] - M[:, 2, 0], M[:, 1, 0] - M[:, 0, 1]
    p, q, r = M[:, 0, 1] + M[:, 1, 0], M[:, 0, 2] + M[:, 2, 0], M[:, 1, 2] + M[:, 2, 1]
    rows = torch.stack([torch.stack(v, 1) for v in ((sq[:, 0], a, b, c), (a, sq[:, 1], p, q), (b, p, sq[:, 2], r),
                                                    (c, q, r, sq[:, 3]))], 1)
    best = rows[torch.arange(M.shape[0], device=M.device), sq.argmax(1)]
    return best / best.norm(dim=1, keepdim=True)


def _surface(g, faces, n):
    """n Gaussians on the faces, as many per face as its area asks, flat along the normal."""
    f = torch.tensor(faces, dtype=torch.float32, device="cuda")
    area = torch.linalg.cross(f[:, 1], f[:, 2]).norm(dim=1)
    which = torch.bucketize(_rand(g, n), torch.cumsum(area / area.sum(), 0)).clamp_(max=f.shape[0] - 1)
    o, u, v, nrm = f[which].unbind(1)
    means = o + _rand(g, n, 1) * u + _rand(g, n, 1) * v
    e1 = u / u.norm(dim=1, keepdim=True)
    e2 = torch.linalg.cross(nrm, e1)
    th = 6.2832 * _rand(g, n, 1)
    t1 = torch.cos(th) * e1 + torch.sin(th) * e2
    quats = _matrix_to_quat(torch.stack([t1, torch.linalg.cross(nrm, t1), nrm], 2))
    ls = (-4.5 + 0.4 * _randn(g, n, 3)).sort(1, descending=True)[0]
    colors = torch.stack([_wave(g, means, 0.0, 1.0, 2.0) for _ in range(3)], 1)
    return [means, ls, quats, torch.sigmoid(1.0 + _randn(g, n)), colors]


def _look(rng, x0, y0, size, w, h):
    """A camera inside the room (90 degrees wide) that looks at a point of one of its walls."""
    lx, ly, lz = size
    c = (x0 + rng.uniform(0.5, lx - 0.5), y0 + rng.uniform(0.5, ly - 0.5), rng.uniform(1.2, 1.8))
    a = rng.uniform(0.05, 0.95)
    wall = rng.choice(((0.0, a * ly), (lx, a * ly), (a * lx, 0.0), (a * lx, ly)))
    return S.look_at(c, (x0 + wall[0], y0 + wall[1], rng.uniform(0.3, lz - 0.3)), w, h, w / 2, w / 2, w / 2, h / 2)


def _scene(case, seed):
    """Gaussians (five tensors), cameras, first row and row count of each view's scene."""
    g, rng = _gen(seed), random.Random(int(seed) * 7919 + 5)
    n, V, w, h = case["n"], case["views"], case["w"], case["h"]
    if case["scene"] == "cloud":
        means = torch.cat([2 * _rand(g, n, 2) - 1, 2 + 4 * _rand(g, n, 1)], 1)
        q = _randn(g, n, 4)
        t = [means, -3.5 + 0.5 * _randn(g, n, 3), q / q.norm(dim=1, keepdim=True), torch.sigmoid(_randn(g, n)), _rand(g, n, 3)]
        cams = [S.look_at((0.1 * k, 0.02 * k, 0.0), (0.1 * k, 0.02 * k + 1e-3, 4.0), w, h, 0.9375 * w, 0.9375 * w, w / 2, h / 2)
                for k in range(V)]
        return t, cams, [0] * V, [n] * V
    if case["scene"] == "room":
        size = (6.0, 5.0, 3.0)
        t = _surface(g, _room(rng, 0.0, 0.0, size, 12), n)
        return t, [_look(rng, 0.0, 0.0, size, w, h) for _ in range(V)], [0] * V, [n] * V
    if case["scene"] == "agents":
        counts = [max(16, a * n // sum(AGENTS)) for a in AGENTS]
        size, parts, cams = (6.0, 5.0, 3.0), [], []
        for c in counts:
            parts.append(_surface(g, _room(rng, 0.0, 0.0, size, 12), c))
            cams += [_look(rng, 0.0, 0.0, size, w, h) for _ in range(V // 8)]
        begin = np.cumsum([0] + counts)[:-1]
        return [torch.cat(p) for p in zip(*parts)], cams, np.repeat(begin, V // 8), np.repeat(counts, V // 8)
    size, parts, cams = (6.567, 7.4, 3.0), [], []      # a 20 x 15 m floor of 3 x 2 rooms, all in every view's scene
    rooms = [(6.667 * i + 0.05, 7.5 * j + 0.05) for i in range(3) for j in range(2)]
    for k, (x0, y0) in enumerate(rooms):
        parts.append(_surface(g, _room(rng, x0, y0, size, 8), n // 6 + (k < n % 6)))
    for k in range(V):
        cams.append(_look(rng, *rooms[k * 6 // V], size, w, h))
    return [torch.cat(p) for p in zip(*parts)], cams, [0] * V, [n] * V


def _image(g, V, C, h, w, lo=0.0, hi=1.0, cell=24.0):
    """Smooth images [V, C, h, w] in [lo, hi], different in every plane."""
    y, x = torch.meshgrid(torch.arange(h, device="cuda") / cell, torch.arange(w, device="cuda") / cell, indexing="ij")
    p = torch.stack([x, y], -1)
    return torch.stack([torch.stack([_wave(g, p, lo, hi, 1.0) for _ in range(C)]) for _ in range(V)])


def _params(case):
    return R.default_params(tile_w=case["tile_w"], tile_h=case["tile_h"], bg=(case["bg"], 0.5 * case["bg"], 0.0))


def _targets(case, seed):
    """Target RGB and depth of a loss, or the three upstream gradients of an autograd call."""
    g = _gen(seed + 500_000)
    V, h, w = case["views"], case["h"], case["w"]
    if case["loss"] == "upstream":
        n = V * h * w
        return [_randn(g, V, 3, h, w) / (3 * n), case["depth_w"] * _randn(g, V, h, w) / n, 0.1 * _randn(g, V, h, w) / n]
    if case["loss"] == "none":
        return []
    return [_image(g, V, 3, h, w), _image(g, V, 1, h, w, 0.5, 5.0)[:, 0].contiguous()]


def _prepare_frame(case, seed):
    t, cams, begin, count = _scene(case, seed)
    g = R.Gaussians(*[x.float().contiguous() for x in t])
    cap = vis = None
    if case["scene"] == "floor":     # most of the floor is behind the camera: capacities from the scene's shape, grown if short
        cap, vis = max(1 << 20, int(0.6 * g.n * case["views"])), max(1 << 16, int(0.4 * g.n * case["views"]))
    pb = R.Problem(np.asarray(begin), np.asarray(count), g.n, case["w"], case["h"], R.cameras_tensor(cams), _params(case),
                   key_capacity=cap, visible_capacity=vis or 0)
    s = {"case": case, "pb": pb, "g": g, "t": _targets(case, seed)}
    img = pb.forward_checked(g, max_retries=4)
    if case["call"] == "autograd":
        s["leaves"] = [getattr(g, k).requires_grad_() for k in FIELDS]
        s["pose"] = torch.zeros(pb.V, 6, device="cuda", requires_grad=True)
        return s
    s["img"], s["loss"] = img, torch.zeros(1, dtype=torch.float64, device="cuda")
    s["d_rgb"], s["d_depth"] = torch.empty_like(img["rgb"]), torch.empty_like(img["depth"])
    if case["loss"] == "ssim":
        s["scratch"] = R.ssim_scratch(pb.V, pb.H, pb.W)
    if case["call"] == "graph":
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _step(s)
        torch.cuda.current_stream().wait_stream(side)
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            s["out"] = _step(s)
    return s


def prepare(case, seed):
    kind = case["kind"]
    if kind == "frame":
        return _prepare_frame(case, seed)
    g = _gen(seed)
    s = {"case": case}
    if kind == "adam":     # a loop that has run for a while: moments in proportion to the gradients
        n = case["n"]
        t = _surface(g, _room(random.Random(seed), 0.0, 0.0, (6.0, 5.0, 3.0), 12), n)
        s["adam"] = R.AdamState(R.Gaussians(*[x.float().contiguous() for x in t]))
        s["grads"] = R.Gaussians(*[1e-7 * _randn(g, *x.shape) for x in t])
        s["adam"].m.copy_(3e-8 * _randn(g, 14 * n))
        s["adam"].v.copy_(1e-14 * (0.5 + _rand(g, 14 * n)))
        s["adam"].step.fill_(100 + seed % 50)
        s["iso"] = torch.zeros(1, dtype=torch.float64, device="cuda")
    elif kind == "loss":
        V, h, w = case["views"], case["h"], case["w"]
        s["rgb_t"] = _image(g, V, 3, h, w)
        s["rgb"] = (s["rgb_t"] + 0.1 * _randn(g, V, 3, h, w)).clamp_(0, 1)
        s["depth_t"] = _image(g, V, 1, h, w, 1.0, 4.0, 90.0)[:, 0].contiguous()
        s["depth"] = s["depth_t"] * (1 + 0.01 * _randn(g, V, h, w))
        s["expo"] = torch.cat([0.1 * _randn(g, V, 1), 0.02 * _randn(g, V, 1)], 1)
        prior = _randn(g, V, 3, h, w) * 0.3
        prior[:, 2] -= 1.0
        s["prior"] = (prior / prior.norm(dim=1, keepdim=True)).contiguous()
        s["cams"] = R.cameras_tensor([_look(random.Random(seed + v), 0.0, 0.0, (6.0, 5.0, 3.0), w, h) for v in range(V)])
        s["scratch"] = R.refine_scratch(V, h, w)
        s["d_rgb"], s["d_depth"], s["d_expo"] = (torch.empty_like(s[k]) for k in ("rgb", "depth", "expo"))
        s["loss"] = torch.zeros(1, dtype=torch.float64, device="cuda")
    elif kind == "pho":
        E, h, w = case["edges"], case["h"], case["w"]
        M = max(2, (E + 1) // 2 * 2)
        rng = np.random.default_rng(seed)
        s["images"] = _image(g, M, 3, h, w)
        s["depths"] = _image(g, M, 1, h, w, 1.5, 4.5, 120.0)[:, 0].contiguous()
        s["depths"][:, : max(1, h // 40)] = 0.0                                # rows without a depth
        cams = []
        for k in range(M):     # the second keyframe of a pair stands a few centimetres beside the first
            if k % 2 == 0:
                c, a = rng.uniform(1.5, 3.5, 3), rng.uniform(0, 2 * math.pi)
            else:
                c, a = c + rng.normal(0, 0.05, 3), a + rng.normal(0, 0.03)
            cams.append(S.look_at(c, c + np.array([math.cos(a), math.sin(a), 0.1]), w, h, w / 2, w / 2, w / 2, h / 2))
        s["cams"] = R.cameras_tensor(cams)
        corr = [(np.array([1.0, *rng.normal(0, 2e-3, 3)]), rng.normal(0, 5e-3, 3), 1 + rng.normal(0, 2e-3)) for _ in range(M)]
        s["corrs"] = R.sim3_tensor(corr)
        s["edges"] = R.pho_edges([(k, k ^ 1, k, k ^ 1, 1.0 + 0.1 * k) for k in range(E)])
        s["pho"] = R.PhoResidual(E)
    else:
        n, V, h, w = case["n"], case["views"], case["h"], case["w"]
        rng = random.Random(seed)
        size, cap = (20.0, 15.0, 3.0), 1 << max(16, math.ceil(math.log2(12 * n + 1)))
        faces = _room(rng, 0.0, 0.0, size, 30)
        s["target"], s["moved"] = ([x.float().contiguous() for x in _surface(g, faces, n)] for _ in range(2))
        s["moved"] = R.Gaussians(*s["moved"])
        s["moved"].means += 0.05 * _randn(g, n, 3)
        s["cams"] = R.cameras_tensor([_look(rng, 0.0, 0.0, size, w, h) for _ in range(V)])
        s["depth"] = _image(g, V, 1, h, w, 0.5, 4.0, 90.0)[:, 0].contiguous()
        s["q"], s["tr"] = (1.0, *(0.01 * rng.gauss(0, 1) for _ in range(3))), tuple(0.05 * rng.gauss(0, 1) for _ in range(3))
        s["occ"], s["free"] = R.VoxSet(cap), R.VoxSet(cap)
        s["out"] = R.Gaussians(*[torch.empty_like(getattr(s["moved"], k)) for k in FIELDS])
    return s


# ------------------------------------------------------------------------------------------
# one pass
# ------------------------------------------------------------------------------------------

def _step(s):
    """One mapping step (or a render) through the stage calls."""
    case, pb, g, img = s["case"], s["pb"], s["g"], s["img"]
    pb.project(g)
    pb.bin_sort()
    wd, d_depth = case["depth_w"], None
    if case["loss"] == "l1_fused":
        d_depth = s["d_depth"] if wd else None
        pb.render_fwd_l1(img, s["t"][0], s["t"][1], 1.0, wd, s["d_rgb"], d_depth, s["loss"])
    else:
        pb.render_fwd(img)
        if case["loss"] == "none":
            return {k: img[k] for k in ("rgb", "depth", "alpha", "last_idx")}
        if case["loss"] == "l1":
            d_depth = s["d_depth"] if wd else None
            R.loss_l1(img["rgb"], s["t"][0], img["depth"], s["t"][1], 1.0, wd, s["d_rgb"], d_depth, s["loss"])
        else:
            R.loss_l1_ssim(img["rgb"], s["t"][0], 0.8, 0.2, s["d_rgb"], s["loss"], s["scratch"])
    grads = pb.render_bwd(g, img, s["d_rgb"], d_depth, None)
    return {"rgb": img["rgb"], "depth": img["depth"], "alpha": img["alpha"], "last_idx": img["last_idx"],
            "loss": s["loss"], "grads": [getattr(grads, k) for k in FIELDS], "pose": pb.pose_grad()}


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "frame":
        if case["call"] == "graph":
            s["graph"].replay()
            return s["out"]
        if case["call"] == "eager":
            return _step(s)
        rgb, depth, alpha = R.rasterize(*s["leaves"], s["pb"], s["pose"])
        got = torch.autograd.grad([rgb, depth, alpha], s["leaves"] + [s["pose"]], s["t"])
        return {"rgb": rgb, "depth": depth, "alpha": alpha, "grads": list(got[:5]), "pose": got[5]}
    if kind == "adam":
        a = s["adam"]
        a.apply(s["grads"], zero_grads=False, iso_weight=case["iso"], iso_loss=s["iso"])
        return {"params": [getattr(a.g, k) for k in FIELDS], "logits": a.logits, "m": a.m, "v": a.v, "iso": s["iso"]}
    if kind == "loss":
        R.loss_refine(s["rgb"], s["rgb_t"], s["expo"], s["depth"], s["depth_t"], 1.75, 0.2, 0.25, s["d_rgb"], s["d_depth"],
                      s["d_expo"], s["loss"], s["scratch"])
        if case["normal"]:
            R.loss_normal(s["depth"], s["prior"], s["cams"], 1e-2, s["d_depth"], s["loss"])
        return {k: s[k] for k in ("loss", "d_rgb", "d_depth", "d_expo")}
    if kind == "pho":
        return s["pho"](s["edges"], s["images"], s["depths"], s["cams"], s["corrs"], stride=case["stride"])
    s["occ"].clear()
    s["occ"].add_boxes(s["target"][0], s["target"][1], 3.0, 0.05)
    s["free"].clear()
    s["free"].add_rays(s["cams"], s["depth"], case["stride"], 0.05)
    m = R.sim3_apply(s["moved"], s["q"], s["tr"], 1.02, s["out"])
    keep = R.dedup_keep(m.means, s["occ"], s["free"], 0.05)
    return {"keep": keep, "moved": [getattr(m, k) for k in FIELDS]}


# ------------------------------------------------------------------------------------------
# the work of one pass
# ------------------------------------------------------------------------------------------

def work(case):
    """Bytes: each input read once, each output written once.  Operations of a render: the (pixel,
    list entry) pairs that a pixel meets before it is opaque, estimated from the scene's shape, at 25
    operations forward and 80 backward each."""
    kind = case["kind"]
    if kind == "frame":
        px = case["views"] * case["w"] * case["h"]
        n = case["n"]
        per = {"cloud": 0.016 * n, "room": 1.6e-4 * n, "agents": 1.6e-4 * n / 6, "floor": 6.5e-5 * n}[case["scene"]]
        pairs = px * min(per, 300.0)
        if case["loss"] == "none":
            return {"bytes": 56 * n + 24 * px, "flops": 25 * pairs}
        return {"bytes": 112 * n + (24 + 16) * px, "flops": 105 * pairs}
    if kind == "adam":
        return {"bytes": 4 * 14 * 7 * case["n"], "flops": 15 * 14 * case["n"]}
    if kind == "loss":
        px = case["views"] * case["w"] * case["h"]
        return {"bytes": (9 * 4 + 3 * 4 + (12 if case["normal"] else 0)) * px, "flops": 3 * (8 * 44 + 60) * px}
    if kind == "pho":
        px = case["edges"] * (case["w"] // case["stride"]) * (case["h"] // case["stride"])
        return {"bytes": 28 * px, "flops": 410 * 0.8 * px}
    rays = case["views"] * (case["w"] // case["stride"]) * (case["h"] // case["stride"])
    return {"bytes": (24 + 112 + 13) * case["n"] + 4 * rays, "flops": 60 * case["n"] + 600 * rays}


# ------------------------------------------------------------------------------------------
# the same in 64 bits
# ------------------------------------------------------------------------------------------

def _x_project(t, cam, xi, w, h, tw, th):
    """EWA projection of all Gaussians into one camera: per visible one mean, conic, opacity, depth and colour, its
    tile rectangle (x0, x1, y0, y1) and its row."""
    mu, ls, q, op, col = t
    Rm, tr, (fx, fy, cx, cy) = cam[:9].view(3, 3), cam[9:12], cam[12:].tolist()
    rho, phi, zero = xi[:3], xi[3:], xi.new_zeros(())
    K = torch.stack([zero, -phi[2], phi[1], phi[2], zero, -phi[0], -phi[1], phi[0], zero]).view(3, 3)
    Rm, tr = Rm + K @ Rm, tr + K @ tr + rho
    row = torch.nonzero((mu.detach() @ Rm.detach()[2] + tr.detach()[2]) > float(np.float32(0.2)))[:, 0]
    mu, ls, q, op, col = (x[row] for x in (mu, ls, q, op, col))
    x, y, z = (mu @ Rm.T + tr).unbind(1)
    qw, qx, qy, qz = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    Rq = torch.stack([1 - 2 * (qy * qy + qz * qz), 2 * (qx * qy - qw * qz), 2 * (qx * qz + qw * qy),
                      2 * (qx * qy + qw * qz), 1 - 2 * (qx * qx + qz * qz), 2 * (qy * qz - qw * qx),
                      2 * (qx * qz - qw * qy), 2 * (qy * qz + qw * qx), 1 - 2 * (qx * qx + qy * qy)], 1).view(-1, 3, 3)
    tx, ty = (x / z).clamp(-0.65 * w / fx, 0.65 * w / fx), (y / z).clamp(-0.65 * h / fy, 0.65 * h / fy)
    o = torch.zeros_like(z)
    J = torch.stack([fx / z, o, -fx * tx / z, o, fy / z, -fy * ty / z], 1).view(-1, 2, 3)
    U = (J @ Rm) @ (Rq * torch.exp(ls)[:, None, :])
    a, b, c = (U[:, 0] ** 2).sum(1) + 0.3, (U[:, 0] * U[:, 1]).sum(1), (U[:, 1] ** 2).sum(1) + 0.3
    det = a * c - b * b
    mx, my = fx * x / z + cx, fy * y / z + cy
    with torch.no_grad():
        mid = 0.5 * (a + c)
        r = torch.ceil(3.0 * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp(min=0))))
        Tx, Ty = -(-w // tw), -(-h // th)
        rect = torch.stack([torch.floor((mx - r) / tw).clamp(0, Tx), (torch.floor((mx + r) / tw) + 1).clamp(0, Tx),
                            torch.floor((my - r) / th).clamp(0, Ty), (torch.floor((my + r) / th) + 1).clamp(0, Ty)], 1).long()
        vis = torch.nonzero((det > 0) & (rect[:, 1] > rect[:, 0]) & (rect[:, 3] > rect[:, 2]))[:, 0]
    feat = torch.stack([mx, my, c / det, -b / det, a / det, op, z, col[:, 0], col[:, 1], col[:, 2]], 1)
    return feat[vis], rect[vis]


def _x_lists(z, rect, tx):
    """Tile lists by depth: the entries' rows, tile by tile, and each tile's first entry and length."""
    nx, cnt = rect[:, 1] - rect[:, 0], (rect[:, 1] - rect[:, 0]) * (rect[:, 3] - rect[:, 2])
    order = torch.sort(z, stable=True)[1]
    row = torch.repeat_interleave(order, cnt[order])
    k = torch.arange(row.numel(), device=row.device) - torch.repeat_interleave(torch.cumsum(cnt[order], 0) - cnt[order], cnt[order])
    tile = (rect[row, 2] + k // nx[row]) * tx + rect[row, 0] + k % nx[row]
    tile, by = torch.sort(tile, stable=True)
    ids, length = torch.unique_consecutive(tile, return_counts=True)
    return row[by], ids, torch.cumsum(length, 0) - length, length


def _x_chunks(length, pix, most=6_000_000):
    """Tiles, longest lists first, in groups that hold at most so many (pixel, entry) pairs."""
    order = torch.argsort(length, descending=True)
    ln = length[order].tolist()
    i = 0
    while i < len(ln):
        k = max(1, most // (pix * max(1, ln[i])))
        yield order[i:i + k], ln[i]
        i += k


def _x_composite(feat, lists, tiles, L, case, px, py):
    """Colour, depth and alpha of a group of tiles' pixels [T, P]."""
    row, _, first, length = lists
    j = torch.arange(L, device=row.device)
    inside = j < length[tiles, None]
    at = row[(first[tiles, None] + j).clamp(max=row.numel() - 1)]
    f = feat.index_select(0, at.view(-1)).view(*at.shape, -1)
    dx, dy = px[:, None, :] - f[..., 0, None], py[:, None, :] - f[..., 1, None]
    sigma = 0.5 * (f[..., 2, None] * dx * dx + f[..., 4, None] * dy * dy) + f[..., 3, None] * dx * dy
    a = (f[..., 5, None] * torch.exp(-sigma)).clamp(max=float(np.float32(0.99)))
    a = torch.where(inside[..., None] & (sigma >= 0) & (a >= float(np.float32(1) / np.float32(255))), a, 0.0)
    T = torch.cumprod(1 - a, 1)
    a = torch.where(T.detach() >= float(np.float32(1e-4)), a, 0.0)     # a pixel stops before the entry that would close it
    T = torch.cumprod(1 - a, 1)
    wgt = a * torch.cat([torch.ones_like(T[:, :1]), T[:, :-1]], 1)
    out = torch.einsum("tlp,tlc->tpc", wgt, f[..., 6:])
    return out[..., 1:] + T[:, -1, :, None] * out.new_tensor([case["bg"], 0.5 * case["bg"], 0.0]).float().double(), out[..., 0], 1 - T[:, -1]


def _x_view(case, t, cam, xi, upstream):
    """Images of one view; with `upstream` (three image gradients) their gradients go into the leaves instead."""
    w, h, tw, th = case["w"], case["h"], case["tile_w"], case["tile_h"]
    tx = -(-w // tw)
    with torch.set_grad_enabled(upstream is not None):
        feat, rect = _x_project(t, cam, xi, w, h, tw, th)
        lists = _x_lists(feat[:, 6].detach(), rect, tx)
        leaf = feat.detach().requires_grad_(upstream is not None)
        rgb = t[0].new_zeros(h * w + 1, 3) + t[0].new_tensor([case["bg"], 0.5 * case["bg"], 0.0]).float().double()
        depth, alpha = t[0].new_zeros(h * w + 1), t[0].new_zeros(h * w + 1)
        p = torch.arange(tw * th, device="cuda")
        for tiles, L in _x_chunks(lists[3], tw * th):
            x = lists[1][tiles, None] % tx * tw + p % tw
            y = lists[1][tiles, None] // tx * th + p // tw
            at = torch.where((x < w) & (y < h), y * w + x, h * w)       # pixels beyond the image: a spare place
            c, d, a = _x_composite(leaf, lists, tiles, L, case, x + 0.5, y + 0.5)
            if upstream is None:
                rgb[at], depth[at], alpha[at] = c, d, a
            else:
                torch.autograd.backward([c, d, a], [u[at] for u in upstream])
        if upstream is None:
            return rgb[:-1].T.reshape(3, h, w), depth[:-1].view(h, w), alpha[:-1].view(h, w)
        if leaf.grad is not None:
            feat.backward(leaf.grad)


def _x_ssim(x, y):
    k = torch.exp(-(torch.arange(11, device="cuda", dtype=torch.float64) - 5) ** 2 / 4.5)
    k = (k / k.sum()).outer(k / k.sum()).view(1, 1, 11, 11)
    x, y = x.reshape(-1, 1, *x.shape[-2:]), y.reshape(-1, 1, *y.shape[-2:])
    mx, my, xx, yy, xy = (F.conv2d(v, k, padding=5) for v in (x, y, x * x, y * y, x * y))
    s = (2 * mx * my + 1e-4) * (2 * (xy - mx * my) + 9e-4) / ((mx * mx + my * my + 1e-4) * (xx - mx * mx + yy - my * my + 9e-4))
    return s.mean()


def _x_frame(case, seed):
    t, cams, begin, count = _scene(case, seed)
    t = [x.float().double().requires_grad_() for x in t]
    cams = R.cameras_tensor(cams).double()
    up = [x.double() for x in _targets(case, seed)]
    V, h, w = case["views"], case["h"], case["w"]
    rows = [[x[int(b):int(b) + int(c)] for x in t] for b, c in zip(begin, count)]
    with torch.no_grad():
        img = [torch.stack(x) for x in zip(*[_x_view(case, rows[v], cams[v], cams.new_zeros(6), None) for v in range(V)])]
    out = {"rgb": img[0], "depth": img[1], "alpha": img[2]}
    if case["loss"] == "none":
        return {**out, "last_idx": None}
    if case["loss"] != "upstream":
        with torch.enable_grad():
            x, d = img[0].clone().requires_grad_(), img[1].clone().requires_grad_()
            if case["loss"] == "ssim":
                loss = sum(0.8 * (x[v] - up[0][v]).abs().mean() + 0.2 * (1 - _x_ssim(x[v], up[0][v])) for v in range(V)) / V
            else:
                loss = (x - up[0]).abs().mean() + float(np.float32(case["depth_w"])) * (d - up[1]).abs().mean()
            gx, gd = torch.autograd.grad(loss, [x, d], allow_unused=True)
        up = [gx, torch.zeros_like(d) if gd is None else gd, torch.zeros_like(d)]
        out |= {"last_idx": None, "loss": loss.detach().view(1)}
    xi = [torch.zeros(6, device="cuda", dtype=torch.float64, requires_grad=True) for _ in range(V)]
    zero = cams.new_zeros(1)
    for v in range(V):
        flat = [torch.cat([up[0][v].reshape(3, -1).T, zero.expand(1, 3)])] + [torch.cat([u[v].reshape(-1), zero]) for u in up[1:]]
        with torch.enable_grad():
            _x_view(case, [x[int(begin[v]):int(begin[v]) + int(count[v])] for x in t], cams[v], xi[v], flat)
    return {**out, "grads": [x.grad for x in t], "pose": torch.stack([x.grad for x in xi])}


def _x_adam(case, seed):
    s = prepare(case, seed)
    a = s["adam"]
    p = [getattr(a.g, k).double() for k in FIELDS]
    gr = [getattr(s["grads"], k).double() for k in FIELDS]
    op = p[3]
    gr[3] = gr[3] * op * (1 - op)
    sc = torch.exp(p[1])
    dev = sc - sc.mean(1, keepdim=True)
    iso = case["iso"] * dev.abs().sum()
    gr[1] = gr[1] + case["iso"] * (torch.sign(dev) - torch.sign(dev).mean(1, keepdim=True)) * sc
    p[3] = a.logits.double()
    gr = torch.cat([x.reshape(-1) for x in gr])
    m = 0.9 * a.m.double() + 0.1 * gr
    v = 0.999 * a.v.double() + 0.001 * gr * gr
    step = int(a.step.item()) + 1
    upd = (m / (1 - 0.9 ** step)) / (torch.sqrt(v / (1 - 0.999 ** step)) + 1e-15)
    out, k = [], 0
    for x, lr in zip(p, a.lr):
        out.append(x - lr * upd[k:k + x.numel()].view_as(x))
        k += x.numel()
    logits, out[3] = out[3], torch.sigmoid(out[3])
    return {"params": out, "logits": logits, "m": m, "v": v, "iso": iso.view(1) if case["iso"] else None}


def _x_normal(depth, prior, cams):
    V, h, w = depth.shape
    x = (torch.arange(w, device="cuda") + 0.5 - cams[:, 14, None]) / cams[:, 12, None]
    y = (torch.arange(h, device="cuda") + 0.5 - cams[:, 15, None]) / cams[:, 13, None]
    P = torch.stack([depth * x[:, None, :], depth * y[:, :, None], depth], 1)
    n = torch.linalg.cross(P[:, :, 2:, 1:-1] - P[:, :, :-2, 1:-1], P[:, :, 1:-1, 2:] - P[:, :, 1:-1, :-2], dim=1)
    return (1 - (n / n.norm(dim=1, keepdim=True) * prior[:, :, 1:-1, 1:-1]).sum(1)).abs().sum() / (V * h * w)


def _x_loss(case, seed):
    s = prepare(case, seed)
    V = case["views"]
    x, d, e = (s[k].double().requires_grad_() for k in ("rgb", "depth", "expo"))
    y, dt = s["rgb_t"].double(), s["depth_t"].double()
    total = 0.0
    for v in range(V):
        z = torch.exp(e[v, 0]) * x[v] + e[v, 1]
        part = (1.75 * (z - y[v]).abs().mean() + float(np.float32(0.2)) * (1 - _x_ssim(z, y[v])) + 0.25 * (d[v] - dt[v]).abs().mean()) / V
        if case["normal"]:
            part = part + float(np.float32(1e-2)) * _x_normal(d[v:v + 1], s["prior"][v:v + 1].double(), s["cams"][v:v + 1].double()) / V
        part.backward()
        total += part.detach()
    return {"loss": total.view(1), "d_rgb": x.grad, "d_depth": d.grad, "d_expo": e.grad}


def _x_quat(q):
    w, x, y, z = q / q.norm()
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z),
                        1 - 2 * (x * x + z * z), 2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x),
                        1 - 2 * (x * x + y * y)]).view(3, 3)


def _x_pho(case, seed):
    s = prepare(case, seed)
    h, w, st, out = case["h"], case["w"], case["stride"], {"cost": [], "H": [], "g": []}
    v, u = torch.meshgrid(torch.arange(0, h, st, device="cuda"), torch.arange(0, w, st, device="cuda"), indexing="ij")
    u, v, delta = u.reshape(-1), v.reshape(-1), 9.0 / 255.0
    for k in range(case["edges"]):
        cs, ct, c1, c2 = s["cams"][k].double(), s["cams"][k ^ 1].double(), s["corrs"][k].double(), s["corrs"][k ^ 1].double()
        d = s["depths"][k, v, u].double()
        p = torch.stack([(u + 0.5 - cs[14]) / cs[12] * d, (v + 0.5 - cs[15]) / cs[13] * d, d], 1)
        x = (p - cs[9:12]) @ cs[:9].view(3, 3)
        x = c1[7] * x @ _x_quat(c1[:4]).T + c1[4:7]
        B = ct[:9].view(3, 3) @ _x_quat(c2[:4]).T / c2[7]
        c = (x - c2[4:7]) @ B.T + ct[9:12]
        iz = 1 / c[:, 2]
        sx, sy = ct[12] * c[:, 0] * iz + ct[14] - 0.5, ct[13] * c[:, 1] * iz + ct[15] - 0.5
        ok = (d > 0) & (c[:, 2] > 0.2) & (sx >= 0) & (sx < w - 1) & (sy >= 0) & (sy < h - 1)
        x, c, iz, sx, sy = x[ok], c[ok], iz[ok], sx[ok], sy[ok]
        x0, y0 = sx.floor().long(), sy.floor().long()
        ax, ay = sx - x0, sy - y0
        I = s["images"][k ^ 1].double()
        i00, i01, i10, i11 = I[:, y0, x0], I[:, y0, x0 + 1], I[:, y0 + 1, x0], I[:, y0 + 1, x0 + 1]
        gx, gy = (i01 - i00) * (1 - ay) + (i11 - i10) * ay, (i10 - i00) * (1 - ax) + (i11 - i01) * ax
        r = s["images"][k][:, v[ok], u[ok]].double() - (i00 + ax * (i01 - i00) + ay * gy)
        a = r.abs()
        om = torch.where(a <= delta, torch.ones_like(a), delta / a)
        rho = torch.where(a <= delta, r * r, delta * (2 * a - delta))
        o = torch.zeros_like(iz)
        P = torch.stack([ct[12] * iz, o, -ct[12] * c[:, 0] * iz * iz, o, ct[13] * iz, -ct[13] * c[:, 1] * iz * iz], 1).view(-1, 2, 3) @ B
        X, Y, Z = x.unbind(1)
        rot = torch.stack([o, Z, -Y, -Z, o, X, Y, -X, o], 1).view(-1, 3, 3)
        A = torch.cat([P, P @ rot, P @ x[:, :, None]], 2)
        J = -(torch.stack([gx, gy], -1)[:, :, None, :] @ A[None])[:, :, 0]
        Sm = torch.einsum("cn,cni,cnj->ij", om, J, J)
        sg = torch.einsum("cn,cni->i", om * r, J)
        scale = (1.0 + 0.1 * k) / max(1, int(ok.sum()))
        out["cost"].append(scale * rho.sum())
        out["H"].append(scale * torch.cat([torch.cat([Sm, -Sm], 1), torch.cat([-Sm, Sm], 1)]))
        out["g"].append(scale * torch.cat([sg, -sg]))
    return {**{k: torch.stack(v) for k, v in out.items()}, "count": None}


def _x_fuse(case, seed):
    s = prepare(case, seed)
    q = torch.tensor(s["q"], dtype=torch.float32, device="cuda").double()
    q = q / q.norm()
    sc, tr = float(np.float32(1.02)), torch.tensor(s["tr"], dtype=torch.float32, device="cuda").double()
    mu, ls, b, op, col = (getattr(s["moved"], k).double() for k in FIELDS)
    (w, x, y, z), (bw, bx, by, bz) = q, b.unbind(1)
    quat = torch.stack([w * bw - x * bx - y * by - z * bz, w * bx + x * bw + y * bz - z * by,
                        w * by - x * bz + y * bw + z * bx, w * bz + x * by - y * bx + z * bw], 1)
    return {"keep": None, "moved": [sc * mu @ _x_quat(q).T + tr, ls + math.log(sc), quat, op, col]}


def exact(case, seed):
    kind = case["kind"]
    if kind == "frame" and case["views"] * case["n"] // (8 if case["scene"] == "agents" else 1) > 12_000_000:
        return None          # the (view, Gaussian) pairs of a fused floor: minutes of 64-bit arithmetic
    return {"frame": _x_frame, "adam": _x_adam, "loss": _x_loss, "pho": _x_pho, "fuse": _x_fuse}[kind](case, seed)
