"""Timed cases: what programs have this package do, through its public calls.

Each case is a dict of plain values; ``listed()`` gives the fixed ones, ``draw``
one more of the same ranges.  Elevations are diamond-square fractals (roughness
0.8, relief 0-1000 m) or noisy tilted planes made on the GPU, with pits and
flats removed by the package's epsilon fill (1e-3 m) as a user's program would
do first; weights are lognormal(0, 1), cotangents N(0, 1).

Kinds:
  dem       flowdir_accumulate: directions and unit counts of one DEM
  counts    accumulate: unit counts of a direction field kept from before
  weighted  weighted_upslope and its backward: areas and the weights' gradient
  batch     BatchPlan.run: many DEMs of uneven sizes in one pipeline
  fill      fill: pits and flats of a raw surface removed
"""
import math
import random

import torch

import paper_1605_05773_gb300 as d8

EPS = 1e-3
KINDS = ("dem", "counts", "weighted", "batch", "fill")


def listed():
    return [
        # a small DEM on its own, as in an interactive tool or a per-basin loop: latency and launches count
        {"name": "dem_512", "kind": "dem", "H": 512, "W": 512, "terrain": "fractal", "rule": "steepest"},
        # the ordinary single raster tile of a survey product
        {"name": "dem_8192", "kind": "dem", "H": 8192, "W": 8192, "terrain": "fractal", "rule": "steepest"},
        # a whole region at once: the largest DEM of the benchmark (4.3 GB of elevations)
        {"name": "dem_32768", "kind": "dem", "H": 32768, "W": 32768, "terrain": "fractal", "rule": "steepest"},
        # smooth engineered or coastal-plain terrain: parallel paths without valleys
        {"name": "plane_8192", "kind": "dem", "H": 8192, "W": 8192, "terrain": "plane", "rule": "steepest"},
        # a study area with holes and an irregular edge, odd sides (rows not aligned), the other direction rule
        {"name": "nodata_3001x5003", "kind": "dem", "H": 3001, "W": 5003, "terrain": "holes", "rule": "lowest_nodata"},
        # the smallest call: counts of a direction field that the program keeps, odd sides
        {"name": "counts_300x257", "kind": "counts", "H": 300, "W": 257, "terrain": "fractal", "strategy": "ring"},
        # one channel through every cell (a terraced or drained field's worst case), by the strategy for long chains
        {"name": "serpentine_8192", "kind": "counts", "H": 8192, "W": 8192, "terrain": "serpentine",
         "strategy": "jump"},
        # rainfall-weighted areas and their gradient: one training step's forward and backward
        {"name": "weighted_8192", "kind": "weighted", "H": 8192, "W": 8192},
        # the same on a small odd raster
        {"name": "weighted_1001x777", "kind": "weighted", "H": 1001, "W": 777},
        # a data set of DEMs of uneven sizes, sides log-uniform in 128..4096, aspect up to 4
        {"name": "batch_512", "kind": "batch", "n": 512, "lo": 128, "hi": 4096},
        # conditioning a raw DEM before use, a large one and a small odd one
        {"name": "fill_8192", "kind": "fill", "H": 8192, "W": 8192, "terrain": "fractal"},
        {"name": "fill_700x933", "kind": "fill", "H": 700, "W": 933, "terrain": "fractal"},
    ]


def _side(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _shape(rng, lo, hi):
    """A side log-uniform in lo..hi, an aspect log-uniform in 1..4, either way round."""
    a = _side(rng, lo, hi)
    b = max(lo, int(round(a / math.exp(rng.uniform(0.0, math.log(4.0))))))
    return (a, b) if rng.random() < 0.5 else (b, a)


def draw(rng):
    kind = rng.choice(KINDS)
    if kind == "batch":
        lo = rng.choice((64, 128, 256))
        return {"kind": kind, "n": _side(rng, 8, 512), "lo": lo, "hi": _side(rng, 2 * lo, 4096)}
    if kind == "dem":
        H, W = _shape(rng, 200, 20000)
        terrain = rng.choice(("fractal", "fractal", "plane", "holes"))
        rule = rng.choice(("steepest", "steepest", "lowest"))
        return {"kind": kind, "H": H, "W": W, "terrain": terrain, "rule": rule + ("_nodata" if terrain == "holes" else "")}
    if kind == "counts":
        H, W = _shape(rng, 200, 16384)
        terrain = rng.choice(("fractal", "fractal", "plane", "serpentine"))
        return {"kind": kind, "H": H, "W": W, "terrain": terrain, "strategy": "jump" if terrain == "serpentine" else "ring"}
    if kind == "weighted":
        H, W = _shape(rng, 200, 10000)
        return {"kind": kind, "H": H, "W": W}
    H, W = _shape(rng, 200, 8192)
    return {"kind": kind, "H": H, "W": W, "terrain": rng.choice(("fractal", "fractal", "plane"))}


# ---- inputs -----------------------------------------------------------------

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _fractal(H, W, gen):
    """Diamond-square on a lattice of squares of a power-of-two side, cropped, rescaled to 0..1000 m."""
    s = 1 << int(math.log2(max(2, min(H, W) - 1)))
    a, b = max(1, -(-(H - 1) // s)), max(1, -(-(W - 1) // s))
    z = torch.empty((a * s + 1, b * s + 1), device="cuda")
    z[::s, ::s] = torch.randn((a + 1, b + 1), generator=gen, device="cuda")
    amp = 1.0
    while s > 1:
        h = s // 2
        amp *= 2.0 ** -0.8
        c = z[0:-1:s, 0:-1:s] + z[s::s, 0:-1:s]
        c += z[0:-1:s, s::s]
        c += z[s::s, s::s]
        c *= 0.25
        c += amp * torch.randn(c.shape, generator=gen, device="cuda")
        z[h::s, h::s] = c
        for along in (0, 1):  # edge midpoints: the two lattice points beside, the one or two centres across
            v, cc = (z, c) if along == 0 else (z.t(), c.t())
            m = v[0::s, 0:-1:s] + v[0::s, s::s]
            m[1:] += cc
            m[:-1] += cc
            m[1:-1] *= 0.25
            m[0] /= 3.0
            m[-1] /= 3.0
            m += amp * torch.randn(m.shape, generator=gen, device="cuda")
            v[0::s, h::s] = m
        del c, m, v, cc
        s = h
    z = z[:H, :W].contiguous()
    lo, hi = z.aminmax()
    return z.sub_(lo).mul_(1000.0 / (hi - lo))


def _plane(H, W, gen):
    i = torch.arange(H - 1, -1, -1, device="cuda", dtype=torch.float32)[:, None]
    j = torch.arange(W - 1, -1, -1, device="cuda", dtype=torch.float32)[None, :]
    return torch.rand((H, W), generator=gen, device="cuda").sub_(0.5).mul_(0.02).add_(0.05 * i + 0.01).add_(0.02 * j)


def _holes(z, gen):
    """NODATA (NaN) outside an irregular study area and in lakes: a few random waves over a threshold."""
    H, W = z.shape
    i = torch.arange(H, device="cuda", dtype=torch.float32)[:, None] / max(H, W)
    j = torch.arange(W, device="cuda", dtype=torch.float32)[None, :] / max(H, W)
    f = torch.zeros_like(z)
    for r in (torch.rand((8, 3), generator=gen, device="cuda").cpu() * 2.0 - 1.0).tolist():
        f += torch.sin(40.0 * (r[0] * i + r[1] * j) + 3.14 * r[2])
    z[f > 3.0] = float("nan")
    return z


def _surface(terrain, H, W, gen):
    return _plane(H, W, gen) if terrain == "plane" else _fractal(H, W, gen)


def _terrain(terrain, H, W, gen):
    z = d8.fill(_surface(terrain, H, W, gen), EPS)
    return _holes(z, gen) if terrain == "holes" else z


def _serpentine(H, W, seed):
    """Boustrophedon direction codes: rows run E and W in turn and step S at their ends; mirrored by the seed."""
    d = torch.empty((H, W), dtype=torch.uint8, device="cuda")
    d[0::2], d[1::2] = 2, 6
    d[0::2, -1], d[1::2, 0] = 4, 4
    if seed & 1:  # left to right
        d = torch.where(d == 2, 6, torch.where(d == 6, 2, d)).to(torch.uint8).flip(1)
    if seed & 2:  # top to bottom
        d = torch.where(d == 4, 0, d).to(torch.uint8).flip(0)
    return d.contiguous()


def _fields(case, seed):
    """Direction field, weights and cotangent of a weighted case."""
    gen = _generator(seed)
    H, W = case["H"], case["W"]
    dirs = d8.flowdir(_terrain("fractal", H, W, gen))
    w = torch.randn((H, W), generator=gen, device="cuda").exp_()
    c = torch.randn((H, W), generator=gen, device="cuda")
    return dirs, w, c


def _shapes(case):
    """A batch's shapes, the same for every seed: the plan is made for them."""
    rng = random.Random(1605)
    return [_shape(rng, case["lo"], case["hi"]) for _ in range(case["n"])]


def _arena(shapes, dtype):
    """One allocation for a batch's outputs, each on a 256-element boundary, and its views."""
    at, views = [], []
    end = 0
    for h, w in shapes:
        at.append(end)
        end += -(-h * w // 256) * 256
    flat = torch.zeros(end, dtype=torch.int32 if dtype == torch.uint32 else dtype, device="cuda")
    for o, (h, w) in zip(at, shapes):
        views.append(flat[o:o + h * w].view(dtype).view(h, w))
    return flat, views


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        gen = _generator(seed)
        shapes = _shapes(case)
        side = 2 * max(max(s) for s in shapes)
        z = _terrain("fractal", side, side, gen)
        # a crop of a pit-free DEM is pit-free: every cell inside it keeps its eight neighbours
        at = (torch.rand((len(shapes), 2), generator=gen, device="cuda").cpu()).tolist()
        zs = []
        for (h, w), (u, v) in zip(shapes, at):
            i, j = int(u * (side - h)), int(v * (side - w))
            zs.append(z[i:i + h, j:j + w].contiguous())
        flat_d, dirs = _arena(shapes, torch.uint8)
        flat_a, counts = _arena(shapes, torch.uint32)
        return {"kind": kind, "plan": d8.BatchPlan(shapes), "zs": zs, "dirs": dirs, "As": counts, "flat_d": flat_d,
                "flat_a": flat_a}
    if kind == "weighted":
        dirs, w, c = _fields(case, seed)
        return {"kind": kind, "dirs": dirs, "w": w.requires_grad_(), "c": c}
    H, W = case["H"], case["W"]
    if kind == "fill":
        return {"kind": kind, "z": _surface(case["terrain"], H, W, _generator(seed))}
    if kind == "counts":
        if case["terrain"] == "serpentine":
            dirs = _serpentine(H, W, seed)
        else:
            dirs = d8.flowdir(_terrain(case["terrain"], H, W, _generator(seed)))
        return {"kind": kind, "dirs": dirs, "strategy": case["strategy"]}
    return {"kind": kind, "z": _terrain(case["terrain"], H, W, _generator(seed)), "rule": case["rule"]}


def run(state):
    kind = state["kind"]
    if kind == "dem":
        dirs, A = d8.flowdir_accumulate(state["z"], state["rule"])
        return {"dir": dirs, "A": A.view(torch.int32)}
    if kind == "counts":
        if state["strategy"] == "ring":
            A = d8.accumulate(state["dirs"])
        else:  # this field's strategy, then back to the default for the program's other rasters
            d8.set_strategy(state["strategy"])
            A = d8.accumulate(state["dirs"])
            d8.set_strategy("ring")
        return {"A": A.view(torch.int32)}
    if kind == "weighted":
        A = d8.weighted_upslope(state["dirs"], state["w"])
        (g,) = torch.autograd.grad(A, state["w"], state["c"])
        return {"A": A.detach(), "dw": g}
    if kind == "batch":
        state["plan"].run(state["zs"], state["dirs"], state["As"])
        return {"dir": state["flat_d"], "A": state["flat_a"]}
    return {"F": d8.fill(state["z"], EPS)}


def work(case):
    """Bytes: each input read once, each output written once.  Operations: eight differences, four scalings
    and eight comparisons a cell for directions, one addition a cell for a sum, three for a relaxed cell."""
    kind = case["kind"]
    if kind == "batch":
        n = sum(h * w for h, w in _shapes(case))
        return {"bytes": 9 * n, "flops": 21 * n}
    n = case["H"] * case["W"]
    if kind == "dem":
        return {"bytes": 9 * n, "flops": 21 * n}
    if kind == "counts":
        return {"bytes": 5 * n, "flops": n}
    if kind == "weighted":
        return {"bytes": 18 * n, "flops": 2 * n}
    return {"bytes": 8 * n, "flops": 9 * n}


# ---- the floating outputs in 64 bits ---------------------------------------

def _downslope(dirs):
    """Flat index of each cell's down-slope cell; H * W where the path ends."""
    H, W = dirs.shape
    di = torch.tensor([-1, -1, 0, 1, 1, 1, 0, -1, 0, 0], device=dirs.device)[dirs.long()]
    dj = torch.tensor([0, 1, 1, 1, 0, -1, -1, -1, 0, 0], device=dirs.device)[dirs.long()]
    i = torch.arange(H, device=dirs.device)[:, None] + di
    j = torch.arange(W, device=dirs.device)[None, :] + dj
    ends = (dirs >= 8) | (i < 0) | (j < 0) | (i >= H) | (j >= W)
    return torch.where(ends, H * W, i * W + j).reshape(-1)


def _path_sums(dirs, w, c):
    """Up-slope sums of w and down-slope path sums of c, by doubling the length of the paths covered."""
    n = dirs.numel()
    end = torch.tensor([n], device=dirs.device)
    to = torch.cat((_downslope(dirs), end))
    A = torch.cat((w.double().reshape(-1), torch.zeros(1, dtype=torch.float64, device=w.device)))
    G = torch.cat((c.double().reshape(-1), torch.zeros(1, dtype=torch.float64, device=w.device)))
    while bool((to < n).any()):
        A = A.index_add(0, to, A)
        A[n] = 0.0
        G = G + G[to]
        to = to[to]
    return A[:n].view(dirs.shape), G[:n].view(dirs.shape)


def _eps_fill(z):
    """The epsilon-fill surface by relaxing every cell at once from above."""
    z = z.double()
    F = torch.full_like(z, float("inf"))
    for edge in (F[0], F[-1], F[:, 0], F[:, -1]):
        edge.fill_(0.0)
    F = torch.where(F == 0.0, z, F)
    inner = z[1:-1, 1:-1]
    while True:
        for _ in range(64):
            rows = torch.minimum(torch.minimum(F[:, :-2], F[:, 1:-1]), F[:, 2:])
            m = torch.minimum(torch.minimum(rows[:-2], rows[1:-1]), rows[2:])
            new = torch.minimum(F[1:-1, 1:-1], torch.where(inner > m, inner, m + EPS))
            same = new == F[1:-1, 1:-1]
            F[1:-1, 1:-1] = new
        if bool(same.all()):
            return F


def exact(case, seed):
    kind = case["kind"]
    if kind == "weighted":
        A, G = _path_sums(*_fields(case, seed))
        return {"A": A, "dw": G}
    if kind == "fill" and case["H"] * case["W"] <= 2_000_000:
        return {"F": _eps_fill(_surface(case["terrain"], case["H"], case["W"], _generator(seed)))}
    return None
