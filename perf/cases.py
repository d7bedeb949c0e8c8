"""Performance cases: what programs that use this library have it do, at the sizes of real use.

A case is a dict of plain values.  `listed()` gives the fixed cases, `draw(rng)` one more of the
same ranges, `prepare(case, seed)` what a program has in hand before the call, `run(state)` one
pass through the public entry points, `work(case)` the bytes and operations a pass cannot do
without, and `exact(case, seed)` what `run` returns, evaluated in 64 bits by the plain formulas
of include/pmc.h with torch alone (none of the library's code).

Kinds of cases:
  frame    reset, then `passes` progressive passes over one frame's shading points, device
           resident (`call` "eager": a call per pass; "graph": one replayed CUDA graph of the
           frame) or from host buffers ("host")
  cast     reset, then per pass the ray caster followed by the pass over its points
  forward  the stand-alone surrogate network over n texture coordinates
  train    training and validation of one surrogate network per material
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2305_07238_gb300 import pmc
from paper_2305_07238_gb300 import workload as W

LEVEL = 10        # 1024 texels per axis, the virtual texture of the library's examples
POS_LEVEL = 6     # voxels of 2^-6 world units (position descriptor)


# ---------------------------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------------------------
def _frame(name=None, nets="mixed", n_mats=64, lo=20, hi=200, sp=0.2, width=1920, height=1080, passes=4,
           cells=1 << 21, entries=8, cost=500, points="frame", offset=0, call="eager", cache=True, surrogates=False):
    """nets: "tiny" (the 8-node example material), "mixed" (n_mats networks of lo..hi nodes, a
    fraction sp of them depending on the shading point) or "deep" (one large UV-only sub-graph per
    network).  points: "frame" (8x8-pixel tiles), "uniform" (UV uniform), "cones" (frame with
    ray-cone footprints, so a mip level per point, shifted by offset), "paths" (direct samples
    and two bounces with visibility classes) or "position" (frame, world-position descriptors on)."""
    case = {"kind": "frame", "nets": nets, "n_mats": n_mats, "lo": lo, "hi": hi, "sp": sp, "width": width,
            "height": height, "passes": passes, "cells": cells, "entries": entries, "cost": cost, "points": points,
            "offset": offset, "call": call, "cache": cache, "surrogates": surrogates}
    return {"name": name, **case} if name else case


def listed():
    return [
        # The smallest use: one 8-node material, 64x64 pixels, a pass per sample.  Latency and launches.
        _frame("tiny_64x64", nets="tiny", n_mats=1, width=64, height=64, cells=8192, cost=0, points="uniform"),
        # An interactive preview at an odd size with a table whose cell count is no power of two.
        _frame("preview_317x179", width=317, height=179, cells=50021),
        # The headline: a 1080p frame of 16 passes replayed as one graph, cost threshold at break-even.
        _frame("frame_1080p", passes=16, call="graph"),
        # The same networks without the cache: plain evaluation of every node of every point.
        _frame("uncached_1080p", passes=2, cache=False),
        # The paper's own rule (and the library's default): every cacheable node looked up and inserted.
        _frame("all_nodes_1080p", cost=0),
        # Many networks of very uneven size (5 to 2000 nodes): short segments beside long programs.
        _frame("uneven_networks_1080p", n_mats=1024, lo=5, hi=2000, cells=1 << 23, passes=2),
        # Path-traced passes, three visibility classes, replacement of less visible entries.
        _frame("paths_640x360", width=640, height=360, cells=1 << 16, cost=0, points="paths"),
        # A frame from host memory: copies in and out are part of the call (an offline renderer).
        _frame("host_1080p", call="host"),
        # Deep networks whose UV-only sub-graph a trained network stands in for.
        _frame("surrogates_1080p", nets="deep", lo=500, hi=2000, passes=2, cost=0, surrogates=True),
        # Primary rays, then the pass with a mip level per point from the ray cones (a renderer's loop).
        {"name": "cast_1080p", "kind": "cast", "n_mats": 64, "lo": 20, "hi": 200, "sp": 0.2, "width": 1920,
         "height": 1080, "passes": 4, "cells": 1 << 21, "entries": 8, "cost": 500, "spheres": 24},
        # The surrogate network by itself, as a program that bakes or previews a material calls it.
        {"name": "forward_1m", "kind": "forward", "n": 1 << 20, "clamp": True},
        # Training the surrogates of a scene's deep materials (the default number of pairs).
        {"name": "train_64", "kind": "train", "n_mats": 64, "lo": 500, "hi": 2000, "n_train": 1 << 16,
         "n_valid": 8192, "epochs": 1},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame"] * 9 + ["cast", "cast", "forward", "forward", "train"])
    width, height = _log(rng, 33, 1920), _log(rng, 17, 1080)
    lo = rng.randint(5, 40)
    common = {"n_mats": _log(rng, 1, 192), "lo": lo, "hi": lo + _log(rng, 10, 400), "sp": rng.choice([0.2, 0.3, 0.4]),
              "passes": rng.randint(1, 6), "width": width, "height": height, "entries": rng.choice([4, 8, 8, 8, 16]),
              "cost": rng.choice([0, 0, 150, 500, 500, 900])}
    cells = max(64, int(width * height * rng.uniform(0.1, 1.5)))
    common["cells"] = 1 << (cells.bit_length() - 1) if rng.random() < 0.7 else cells
    if kind == "cast":
        return {"kind": "cast", "spheres": rng.randint(0, 48), **common}
    if kind == "forward":
        return {"kind": "forward", "n": _log(rng, 100, 3_000_000), "clamp": rng.random() < 0.7}
    if kind == "train":
        return {"kind": "train", "n_mats": rng.randint(3, 96), "lo": 60, "hi": rng.randint(200, 900),
                "n_train": 1 << rng.randint(9, 15), "n_valid": rng.randint(1000, 8192), "epochs": rng.randint(1, 2)}
    what = rng.choice(["frame", "frame", "frame", "uniform", "cones", "paths", "position", "uncached", "surrogates"])
    call = rng.choice(["eager", "eager", "graph", "graph", "host"])
    if what == "uncached":
        return _frame(**common, cache=False, call=call)
    if what == "surrogates":
        common.update(n_mats=min(common["n_mats"], 48), lo=60, hi=rng.randint(200, 900), cost=0)
        return _frame(**common, nets="deep", call=call, surrogates=True)
    return _frame(**common, points=what, call=call, offset=rng.choice([0, -1]) if what == "cones" else 0)


# ---------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=4)
def _networks(nets, n_mats, lo, hi, sp):
    """The scene's networks: the same for every view (seed) of it."""
    if nets == "tiny":
        return [W.material_tiny()]
    if nets == "deep":
        return W.surrogate_materials(n_mats, lo, hi, seed=0)
    return W.random_materials(n_mats, lo, hi, sp, seed=0)


def _theta(rng):
    """Parameters of one surrogate network at the scale training starts from: weights uniform
    with the He bound, small biases, the output near the middle of [0, 1]."""
    th = np.zeros(pmc.MLP_PARAMS, dtype=np.float32)
    b = math.sqrt(6.0 / 64.0)
    th[:4096] = rng.uniform(-b, b, 4096)
    th[4096:4160] = rng.uniform(-0.1, 0.1, 64)
    th[4160:8256] = rng.uniform(-b, b, 4096)
    th[8256:8320] = rng.uniform(-0.1, 0.1, 64)
    th[8320:8512] = rng.uniform(-b, b, 192) * 0.3
    th[8512:] = 0.5
    return th


def _thetas(case, seed):
    rng = np.random.default_rng([seed, 21])
    return [_theta(rng) for _ in range(case["n_mats"])]


def _points(case, seed):
    """The passes' shading points as dicts of device tensors."""
    w, h, k = case["width"], case["height"], case["passes"]
    if case["points"] == "uniform":
        pts = W.points_uniform(w * h * k, seed=seed, n_mats=case["n_mats"])
        return [pmc.points_to_device(W.slice_points(pts, p * w * h, (p + 1) * w * h)) for p in range(k)]
    frame = W.Frame(W.FrameSpec(width=w, height=h, n_mats=case["n_mats"], seed=seed))
    if case["points"] == "paths":
        return [pmc.points_to_device(frame.points_paths(p)) for p in range(k)]
    if case["points"] == "cones":
        return [pmc.points_to_device(frame.points(p, cones=True)) for p in range(k)]
    return [frame.points_torch(p) for p in range(k)]


def _cache(case, mats):
    flags = 0 if case.get("cache", True) else pmc.PMC_CACHE_OFF
    points = case.get("points", "cast")
    if points == "paths":
        flags |= pmc.PMC_REPLACE_VISIBILITY
    if points == "position":
        flags |= pmc.PMC_POSITION_DESCRIPTOR
    return pmc.Cache(mats, n_cells=case["cells"], n_entries=case["entries"], uv_level=LEVEL, flags=flags,
                     level_offset=case.get("offset", 0), pos_level=POS_LEVEL, min_root_cost=case["cost"])


def _pinned(a):
    t = torch.empty(a.shape, dtype=a.dtype, pin_memory=True)
    t.copy_(a)
    return t.numpy()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "forward":
        g = torch.Generator(device="cuda").manual_seed(seed)
        uv = torch.rand((2, case["n"]), generator=g, device="cuda")
        return {"case": case, "theta": torch.from_numpy(_theta(np.random.default_rng([seed, 21]))).cuda(),
                "u": uv[0].contiguous(), "v": uv[1].contiguous()}
    if kind == "train":
        mats = _networks("deep", case["n_mats"], case["lo"], case["hi"], 0.2)
        return {"case": case, "seed": seed, "cache": pmc.Cache(mats, n_cells=4096, n_entries=8, uv_level=LEVEL)}
    mats = _networks(case.get("nets", "mixed"), case["n_mats"], case["lo"], case["hi"], case["sp"])
    cache = _cache(case, mats)
    if kind == "cast":
        scene = W.Scene(W.SceneSpec(n_mats=case["n_mats"], n_spheres=case["spheres"], width=case["width"],
                                    height=case["height"], seed=seed))
        n = case["width"] * case["height"]
        pts = pmc.cast_rays(scene.objects, scene.camera, seed, 0)
        sizes = [n] * case["passes"]
        state = {"scene": scene, "pts": pts, "seed": seed}
    else:
        passes = _points(case, seed)
        sizes = [int(p["u"].numel()) for p in passes]
        state = {"passes": passes}
    if case.get("surrogates"):
        for m, th in enumerate(_thetas(case, seed)):
            cache.set_surrogate(m, th)
    rgb = [torch.empty((3, n), dtype=torch.float32, device="cuda") for n in sizes]
    hits = [torch.empty(n, dtype=torch.int16, device="cuda") for n in sizes]
    if case.get("call") == "host":
        state["passes"] = [{k: _pinned(t).view(np.uint32) if k == "mat" else _pinned(t) for k, t in p.items()}
                           for p in passes]
        rgb = [torch.empty((3, n), dtype=torch.float32, pin_memory=True).numpy() for n in sizes]
        hits = [torch.empty(n, dtype=torch.int16, pin_memory=True).numpy() for n in sizes]
    elif case.get("call") == "graph":
        # the first pass of a size allocates the cache's scratch, so it runs before the recording
        cache.eval_batch(passes[0], rgb[0], hits[0])
        state["graph"] = cache.graph(passes, rgb, hits, reset=True)
    return {"case": case, "cache": cache, "rgb": rgb, "hits": hits, **state}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "forward":
        return pmc.mlp_forward(state["theta"], state["u"], state["v"], clamp=case["clamp"])
    cache = state["cache"]
    if kind == "train":
        rmse = cache.train_surrogates(n_train=case["n_train"], n_valid=case["n_valid"], epochs=case["epochs"],
                                      seed=state["seed"])
        return {"rmse": rmse, "theta": np.stack([cache.get_surrogate(m)["theta"] for m in range(case["n_mats"])])}
    rgb, hits = state["rgb"], state["hits"]
    if "graph" in state:
        state["graph"].launch()
        return {"rgb": rgb, "hits": hits}
    cache.reset()
    if kind == "cast":
        scene, pts = state["scene"], state["pts"]
        for p in range(case["passes"]):
            pmc.cast_rays(scene.objects, scene.camera, state["seed"], p, out=pts)
            cache.eval_batch(pts, rgb[p], hits[p])
        return {"rgb": rgb, "hits": hits, "points": pts}
    if case["call"] == "host":
        cache.eval_passes_host(state["passes"], rgb, hits)
    else:
        for p, pts in enumerate(state["passes"]):
            cache.eval_batch(pts, rgb[p], hits[p])
    return {"rgb": rgb, "hits": hits}


# ---------------------------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------------------------
MLP_FLOPS = 2 * (64 * 64 + 64 * 64 + 64 * 3)


def _costs(mats, case):
    """Mean operations of one point: all nodes, and the nodes outside cacheable sub-graphs."""
    full, outer = [], []
    for nodes in mats:
        a = _analyse(nodes, case["cost"], case.get("points") == "position")
        n = len(nodes)
        need = [False] * n
        need[n - 1] = n - 1 not in a["roots"]
        for i in range(n - 1, -1, -1):
            if need[i]:
                for j in a["inp"][i]:
                    if j not in a["roots"]:
                        need[j] = True
        full.append(sum(c for c, r in zip(a["cost"], a["reach"]) if r))
        outer.append(sum(c for c, r in zip(a["cost"], need) if r))
    return float(np.mean(full)), float(np.mean(outer))


def work(case):
    kind = case["kind"]
    if kind == "forward":
        return {"bytes": case["n"] * 20 + 4 * pmc.MLP_PARAMS, "flops": case["n"] * MLP_FLOPS}
    if kind == "train":
        mats = _networks("deep", case["n_mats"], case["lo"], case["hi"], 0.2)
        evaluate, _ = _costs(mats, {"cost": 0})
        pairs = case["n_mats"] * (case["n_train"] * case["epochs"] * 3 + case["n_valid"])
        samples = case["n_mats"] * (case["n_train"] + case["n_valid"])
        return {"bytes": 4 * case["n_mats"] * pmc.MLP_PARAMS, "flops": pairs * MLP_FLOPS + samples * evaluate}
    mats = _networks(case.get("nets", "mixed"), case["n_mats"], case["lo"], case["hi"], case["sp"])
    full, outer = _costs(mats, case)
    points, passes = case.get("points", "cast"), case["passes"]
    n = case["width"] * case["height"]
    if points == "paths":
        n += int(round(0.5 * n)) + int(round(0.25 * n))
    per_point = 36 + 14 + (1 if points == "paths" else 16 if points in ("cones", "cast") else 0)
    if case.get("surrogates"):
        flops = n * passes * (outer + MLP_FLOPS)
    elif not case.get("cache", True):
        flops = n * passes * full
    else:   # the first pass evaluates everything; later ones at least what depends on the shading point
        flops = n * (full + (passes - 1) * outer)
    return {"bytes": n * passes * per_point, "flops": flops}


# ---------------------------------------------------------------------------------------------
# The same in 64 bits: the node formulas, the descriptors and the keep-first table of
# include/pmc.h, with torch on whole batches of points
# ---------------------------------------------------------------------------------------------
M32 = 0xFFFFFFFF


def _node_cost(op, ip0):
    """The node cost model of include/pmc.h."""
    return {W.OP_UV_AFFINE: 8, W.OP_FBM: 4 + 47 * ip0, W.OP_VORONOI: 99, W.OP_CHECKER: 4, W.OP_RAMP: 23,
            W.OP_MIX: 17, W.OP_ADD: 9, W.OP_MUL: 9, W.OP_POW: 18, W.OP_FACING: 8}.get(op, 0)


def _inputs(nodes):
    return [[j for j in row if j >= 0] for row in nodes["inp"].tolist()]


def _below(inp, i):
    """The nodes of i's sub-graph, i among them."""
    seen, todo = {i}, [i]
    while todo:
        for j in inp[todo.pop()]:
            if j not in seen:
                seen.add(j)
                todo.append(j)
    return seen


def _analyse(nodes, min_cost, pos_desc):
    """Reachable nodes, and the cacheable ones: {node: 1 for a UV, 2 for a position descriptor}, the
    operations of their sub-graphs, and whether another cacheable node is among them."""
    n = len(nodes)
    op = nodes["op"].tolist()
    inp = _inputs(nodes)
    cost = [_node_cost(o, ip) for o, ip in zip(op, nodes["ip"][:, 0].tolist())]
    reach = [False] * n
    reach[-1] = True
    for i in range(n - 1, -1, -1):
        if reach[i]:
            for j in inp[i]:
                reach[j] = True
    const, uv, pos, sp = 0, 1, 2, 3
    cls = []
    for i in range(n):
        if op[i] == W.OP_UV:
            c = uv
        elif op[i] == W.OP_POSITION:
            c = pos if pos_desc else sp
        elif op[i] == W.OP_NORMAL:
            c = sp
        else:
            kinds = {cls[j] for j in inp[i]} - {const}
            c = const if not kinds else kinds.pop() if len(kinds) == 1 else sp
        cls.append(c)
    feeds_sp = [False] * n
    for i in range(n):
        if reach[i] and cls[i] == sp:
            for j in inp[i]:
                feeds_sp[j] = True
    inputs = (W.OP_UV, W.OP_POSITION, W.OP_NORMAL, W.OP_CONST)
    roots, below, nested = {}, {}, {}
    for i in range(n):
        if not reach[i] or cls[i] not in (uv, pos) or op[i] in inputs or not (i == n - 1 or feeds_sp[i]):
            continue
        seen = _below(inp, i)
        if sum(op[j] not in inputs for j in seen) >= 2 and sum(cost[j] for j in seen) >= min_cost:
            below[i] = sum(cost[j] for j in seen)
            nested[i] = any(j in roots for j in seen)
            roots[i] = cls[i]
    return {"reach": reach, "inp": inp, "cost": cost, "roots": roots, "below": below, "nested": nested}


def _mul32(x, c):
    return (x * c) & M32


def _lattice(i, j, seed):
    h = _mul32(i & M32, 73856093) ^ _mul32(j & M32, 19349663) ^ ((seed * 83492791) & M32)
    h = h ^ (h >> 16)
    h = _mul32(h, 0x85EBCA6B)
    h = h ^ (h >> 13)
    h = _mul32(h, 0xC2B2AE35)
    return h ^ (h >> 16)


def _noise(x, y, seed):
    """Gradient noise on the 8 unit gradients at multiples of 45 degrees, quintic fade."""
    x0, y0 = torch.floor(x), torch.floor(y)
    fx, fy = x - x0, y - y0
    di = torch.tensor([[0], [1], [0], [1]], device=x.device)
    dj = torch.tensor([[0], [0], [1], [1]], device=x.device)
    g = _lattice(x0.long() + di, y0.long() + dj, seed) & 7
    ang = torch.tensor([math.pi / 4 * k for k in range(8)], dtype=torch.float64, device=x.device)
    d = torch.cos(ang)[g] * (fx - di) + torch.sin(ang)[g] * (fy - dj)
    sx = fx ** 3 * (fx * (fx * 6 - 15) + 10)
    sy = fy ** 3 * (fy * (fy * 6 - 15) + 10)
    a = d[0] + sx * (d[1] - d[0])
    b = d[2] + sx * (d[3] - d[2])
    return a + sy * (b - a)


def _voronoi(x, y, scale, seed):
    x, y = x * scale, y * scale
    x0, y0 = torch.floor(x), torch.floor(y)
    k = torch.arange(9, device=x.device).reshape(9, 1)
    di, dj = k % 3 - 1, k // 3 - 1
    h = _lattice(x0.long() + di, y0.long() + dj, seed)
    px = di + 0.25 + 0.5 * (h & 0xFFFF) / 65536.0
    py = dj + 0.25 + 0.5 * (h >> 16) / 65536.0
    return torch.sqrt(((px - (x - x0)) ** 2 + (py - (y - y0)) ** 2).amin(dim=0))


def _evaluate(nd, a, pt):
    """One node for all points: a = its inputs' values (each 3 tensors), pt = u, v, position, normal."""
    op, fp, ip = int(nd["op"]), [float(x) for x in nd["fp"]], [int(x) for x in nd["ip"]]
    one = torch.ones_like(pt["u"])
    if op == W.OP_UV:
        return [pt["u"], pt["v"], 0 * one]
    if op == W.OP_POSITION:
        return [pt["px"], pt["py"], pt["pz"]]
    if op == W.OP_NORMAL:
        return [pt["nx"], pt["ny"], pt["nz"]]
    if op == W.OP_CONST:
        return [fp[0] * one, fp[1] * one, fp[2] * one]
    if op == W.OP_UV_AFFINE:
        x, y = a[0][0], a[0][1]
        return [fp[0] * x + fp[1] * y + fp[4], fp[2] * x + fp[3] * y + fp[5], 0 * one]
    if op == W.OP_FBM:
        total, amp, freq, norm = 0 * one, 1.0, fp[0], 0.0
        for k in range(ip[0]):
            total = total + amp * _noise(a[0][0] * freq, a[0][1] * freq, ip[1] + k)
            norm, amp, freq = norm + amp, amp * fp[2], freq * fp[1]
        r = [0.5 + total / norm] * 3
    elif op == W.OP_VORONOI:
        r = [_voronoi(a[0][0], a[0][1], fp[0], ip[1])] * 3
    elif op == W.OP_CHECKER:
        even = torch.remainder(torch.floor(a[0][0] * fp[0]) + torch.floor(a[0][1] * fp[0]), 2.0) == 0
        r = [torch.where(even, fp[1 + c] * one, fp[4 + c] * one) for c in range(3)]
    elif op == W.OP_RAMP:
        t, ns = a[0][0].clamp(0, 1), ip[0]
        r = []
        for c in range(3):
            col = [fp[4 + 3 * k + c] for k in range(ns)]
            v = col[0] * one
            for k in range(ns - 1):
                if fp[k + 1] > fp[k]:
                    f = (t - fp[k]) / (fp[k + 1] - fp[k])
                    v = torch.where(t >= fp[k], col[k] + (col[k + 1] - col[k]) * f, v)
            v = torch.where(t >= fp[ns - 1], col[-1] * one, v)
            r.append(torch.where(t <= fp[0], col[0] * one, v))
    elif op == W.OP_MIX:
        f = (a[2][0] if len(a) > 2 else fp[0] * one).clamp(0, 1)
        r = [x + (y - x) * f for x, y in zip(a[0], a[1])]
    elif op == W.OP_ADD:
        r = [x + y for x, y in zip(a[0], a[1])]
    elif op == W.OP_MUL:
        r = [x * y for x, y in zip(a[0], a[1])]
    elif op == W.OP_POW:
        r = [x.clamp(min=0) ** fp[0] for x in a[0]]
    else:   # FACING
        r = [(a[0][0] * fp[0] + a[0][1] * fp[1] + a[0][2] * fp[2]).abs()] * 3
    return [x.clamp(0, 1) for x in r]


def _signed(c):
    return c - (1 << 64) if c >= 1 << 63 else c


def _shr(z, k):
    return (z >> k) & ((1 << (64 - k)) - 1)


def _address(key, n_cells):
    """The cell (SplitMix64's output function modulo the cells) and the check value (the upper
    half of MurmurHash3's 64-bit finaliser; 0 reads 1) of a descriptor."""
    z = (key ^ _shr(key, 30)) * _signed(0xBF58476D1CE4E5B9)
    z = (z ^ _shr(z, 27)) * _signed(0x94D049BB133111EB)
    z = z ^ _shr(z, 31)
    cell = (torch.remainder(_shr(z, 1), n_cells) * 2 + (z & 1)) % n_cells
    z = key ^ _signed(0x9E3779B97F4A7C15)
    z = (z ^ _shr(z, 33)) * _signed(0xFF51AFD7ED558CCD)
    z = (z ^ _shr(z, 33)) * _signed(0xC4CEB9FE1A85EC53)
    h2 = _shr(z ^ _shr(z, 33), 32)
    return cell, torch.where(h2 == 0, torch.ones_like(h2), h2)


def _key(case, m, node, kind, p):
    if kind == 2:
        vox = [torch.floor((p[c] * 2.0 ** POS_LEVEL).clamp(-512, 511)).long() + 512 for c in ("px", "py", "pz")]
        return (m << 48) | (node << 32) | (1 << 31) | (vox[0] << 20) | (vox[1] << 10) | vox[2]
    if "g1u" in p:
        s = torch.minimum(p["g1u"] * p["g1u"] + p["g1v"] * p["g1v"], p["g2u"] * p["g2u"] + p["g2v"] * p["g2v"])
        frac, e = torch.frexp(s)          # s = (2 frac) 2^(e - 1), frac in [1/2, 1)
        e = e.long() - 1
        level = torch.where(frac == 0.5, -((e + 1) >> 1), -((e + 2) >> 1)) + case["offset"]
        level = torch.where(s == 0, torch.full_like(level, 13), level).clamp(0, 13)
    else:
        level = torch.full_like(p["u"], LEVEL, dtype=torch.int64)
    res = torch.ones_like(level) << level
    t = [torch.minimum(torch.floor(p[c].clamp(0, 1).double() * res).long(), res - 1) for c in ("u", "v")]
    return (m << 48) | (node << 32) | (level << 26) | (t[0] << 13) | t[1]


def _sources(case, word, when, order):
    """For every probe, the probe whose value it reads from the keep-first table, or -1 (a miss).
    word: cell and check value, when: pass, order: position in its pass.  A pass sees the entries of
    earlier ones; then the first miss of each word enters while its cell has an empty entry."""
    src = torch.full_like(word, -1)
    words, ids = word[:0], word[:0]
    used = torch.zeros(case["cells"], dtype=torch.int64, device=word.device)
    for k in range(case["passes"]):
        probe = (when == k).nonzero().flatten()
        if len(words) and len(probe):
            at = torch.searchsorted(words, word[probe]).clamp(max=len(words) - 1)
            hit = words[at] == word[probe]
            src[probe[hit]] = ids[at[hit]]
            probe = probe[~hit]
        by = probe[torch.argsort(order[probe])]
        by = by[torch.argsort(word[by], stable=True)]
        new = torch.ones_like(by, dtype=torch.bool)
        new[1:] = word[by][1:] != word[by][:-1]
        by = by[new]
        by = by[torch.argsort(order[by])]
        cell, perm = torch.sort(_shr(word[by], 32), stable=True)
        by = by[perm]
        at = torch.arange(len(by), device=by.device)
        start = torch.ones_like(by, dtype=torch.bool)
        start[1:] = cell[1:] != cell[:-1]
        rank = at - torch.cummax(torch.where(start, at, torch.zeros_like(at)), dim=0).values if len(by) else at
        ok = rank + used[cell] < case["entries"]
        used += torch.bincount(cell[ok], minlength=case["cells"])
        words, perm = torch.sort(torch.cat([words, word[by[ok]]]))
        ids = torch.cat([ids, by[ok]])[perm]
    return src


def _mlp(theta, u, v):
    """sin/cos features of half-range frequencies 1..16, two hidden layers of 64, 3 outputs."""
    th = torch.as_tensor(theta, device=u.device).double()
    k = math.pi * torch.arange(1, 17, dtype=torch.float64, device=u.device)
    x = torch.cat([f(c.double()[:, None] * k) for c in (u, v) for f in (torch.sin, torch.cos)], dim=1)
    x = torch.relu(x @ th[:4096].reshape(64, 64) + th[4096:4160])
    x = torch.relu(x @ th[4160:8256].reshape(64, 64) + th[8256:8320])
    return x @ th[8320:8512].reshape(64, 3) + th[8512:]


def _exact_frame(case, seed):
    mats = _networks(case["nets"], case["n_mats"], case["lo"], case["hi"], case["sp"])
    passes = _points(case, seed)
    thetas = _thetas(case, seed) if case["surrogates"] else None
    plans = [_analyse(nodes, case["cost"], case["points"] == "position") for nodes in mats]
    sizes = [len(p["u"]) for p in passes]
    pts = {f: torch.cat([p[f] for p in passes]) for f in passes[0]}
    when = torch.cat([torch.full((n,), k, device=pts["u"].device) for k, n in enumerate(sizes)])
    local = torch.cat([torch.arange(n, device=pts["u"].device) for n in sizes])
    of_mat = [(pts["mat"] == m).nonzero().flatten() for m in range(len(mats))]
    # which probes read which values: a matter of descriptors alone
    base, word, order, pass_of, total = {}, [], [], [], 0
    learned = [None] * len(mats)
    for m, plan in enumerate(plans):
        idx = of_mat[m]
        if thetas:   # a surrogate takes the costliest cacheable node that reads no other one
            top = [(-plan["below"][r], r) for r in plan["roots"] if not plan["nested"][r]]
            learned[m] = min(top)[1] if top else None
        if not case["cache"]:
            continue
        p = {f: t[idx] for f, t in pts.items()}
        for r, kind in plan["roots"].items():
            if r == learned[m]:
                continue
            cell, h2 = _address(_key(case, m, r, kind, p), case["cells"])
            base[m, r] = total
            total += len(idx)
            word.append((cell << 32) | h2)
            order.append((local[idx] << 16) | r)
            pass_of.append(when[idx])
    paths = case["points"] == "paths"   # which entries a later pass replaces is a sequential rule of its own
    if total and not paths:
        src = _sources(case, torch.cat(word), torch.cat(pass_of), torch.cat(order))
    elif total:
        src = torch.full((total,), -1, device=when.device)
    values = torch.zeros((total, 3), dtype=torch.float64, device=when.device)
    out = torch.zeros((3, len(when)), dtype=torch.float64, device=when.device)
    hits = torch.zeros(len(when), dtype=torch.int64, device=when.device)
    # a second sweep settles values read from a later network's entry (equal words of two descriptors)
    for sweep in range(2 if total else 1):
        for m, (nodes, plan) in enumerate(zip(mats, plans)):
            idx = of_mat[m]
            if not len(idx):
                continue
            pt = {f: t[idx].double() for f, t in pts.items()}
            need = [False] * len(nodes)
            need[-1] = True
            last = {}
            for i in range(len(nodes) - 1, -1, -1):
                if need[i] and i != learned[m]:
                    for j in plan["inp"][i]:
                        need[j] = True
                        last.setdefault(j, i)
            val = {}
            for i, nd in enumerate(nodes):
                if not need[i]:
                    continue
                if i == learned[m]:
                    val[i] = list(_mlp(thetas[m], pt["u"], pt["v"]).clamp(0, 1).T)
                else:
                    val[i] = _evaluate(nd, [val[j] for j in plan["inp"][i]], pt)
                if (m, i) in base:
                    b = base[m, i]
                    s = src[b:b + len(idx)]
                    values[b:b + len(idx)] = torch.stack(val[i], dim=1).float().double()
                    stored = values[s.clamp(min=0)]
                    val[i] = [torch.where(s >= 0, stored[:, c], val[i][c]) for c in range(3)]
                    if sweep == 0:
                        hits[idx] += s >= 0
                for j in set(plan["inp"][i]):
                    if last.get(j) == i:
                        del val[j]
            out[:, idx] = torch.stack(val[len(nodes) - 1])
    rgb = [x.contiguous() for x in torch.split(out, sizes, dim=1)]
    hits = [x.short() for x in torch.split(hits, sizes)]
    if paths:
        rgb[1:], hits[1:] = [None] * (len(sizes) - 1), [None] * (len(sizes) - 1)
    return {"rgb": rgb, "hits": hits}


def exact(case, seed):
    """None where there is no such value or it takes too long: a caster's pixels at object edges
    depend on FP32 rounding, and trained parameters on the BF16 rounding of every step before."""
    if case["kind"] == "forward":
        g = torch.Generator(device="cuda").manual_seed(seed)
        uv = torch.rand((2, case["n"]), generator=g, device="cuda")
        y = _mlp(_theta(np.random.default_rng([seed, 21])), uv[0], uv[1]).T
        return y.clamp(0, 1) if case["clamp"] else y
    if case["kind"] != "frame" or case["n_mats"] * (case["lo"] + case["hi"]) > 200_000:
        return None
    return _exact_frame(case, seed)
