"""The work that users of this framework have it do, as timed cases.

A case is one call (or one step made of the calls a program makes together)
through the public entry points of ``paper_1805_08500_gb300``:

  map      one shortest-path map into device buffers (``Scene.compute``)
  host     the same map into page-locked host buffers (``spm_compute_host``)
  frame    sources moved on the device, the map, the agents' mean distance
  grad     the differentiable step: ``agent_loss`` and its backward
  batch    many scenes together (``spm_batch_compute``)
  paths    shortest paths walked back from points of a computed map

Scenes come from ``scenegen``: rectangles, random convex polygons, mazes and
the paper's rows of squares. ``tuning`` names the workload class whose culling
settings the program takes at set-up (``Scene.autotune(cache_key=...)``, from
the committed cache, as the benchmark does); "" keeps the library's defaults.
"""
import math

import numpy as np
import torch

import paper_1805_08500_gb300 as spm
import scenegen as sg


SIDES = (128, 256, 512, 1024)  # grid sides of a batch's scenes
PATH_CAP = 256                 # points of a path that are kept

# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # smallest map: a few rectangles, one source, where launches count
        {"name": "map_rects256", "kind": "map", "scene": "rects", "n": 256, "polys": 8, "points": 1, "segs": 0,
         "tuning": "rects256"},
        # the paper's Table 2 scene (64 squares, 256 vertices) at its own 1000^2 grid
        {"name": "map_squares64", "kind": "map", "scene": "squares", "n": 1000, "k": 8, "tuning": "profiling64"},
        # ordinary obstacles and sources, the settings a user gets without tuning
        {"name": "map_polys512_untuned", "kind": "map", "scene": "polys", "n": 512, "pitch": 4, "polys": 60,
         "points": 2, "segs": 1, "tuning": ""},
        # the benchmark's polygon scene, tuned
        {"name": "map_polys1024", "kind": "map", "scene": "polys", "n": 1024, "pitch": 4, "polys": 200,
         "points": 3, "segs": 2, "tuning": "polys1024"},
        # an odd grid: rows that are no multiple of a tile or of a vector store
        {"name": "map_polys1501_odd", "kind": "map", "scene": "polys", "n": 1501, "pitch": 4, "polys": 240,
         "points": 2, "segs": 1, "tuning": "diff2048_grad"},
        # the headline: a deep maze at the largest grid
        {"name": "map_maze4096", "kind": "map", "scene": "maze", "cells": 64, "cell": 256, "n": 4096, "points": 4,
         "tuning": "maze4096"},
        # a program that keeps the field on the host
        {"name": "host_polys1024", "kind": "host", "scene": "polys", "n": 1024, "pitch": 4, "polys": 200,
         "points": 3, "segs": 2, "tuning": "polys1024"},
        # a crowd's frame: the sources have moved, the field and the agents' mean follow
        {"name": "frame_maze2048", "kind": "frame", "scene": "maze", "cells": 32, "cell": 256, "n": 2048,
         "points": 4, "agents": 100000, "tuning": "maze2048"},
        # the differentiable step of the benchmark: loss and gradients of 100k agents
        {"name": "grad_polys2048", "kind": "grad", "scene": "polys", "n": 2048, "pitch": 4, "polys": 150,
         "points": 4, "segs": 1, "agents": 100000, "tuning": "diff2048_grad"},
        # many scenes in one launch sequence, as many of each grid side
        {"name": "batch_64", "kind": "batch", "each": 16, "poly_lo": 10, "poly_hi": 300},
        # navigation queries on a finished map
        {"name": "paths_polys1024", "kind": "paths", "scene": "polys", "n": 1024, "pitch": 4, "polys": 200,
         "points": 3, "segs": 2, "queries": 32, "tuning": "polys1024"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_polys(rng, lo, hi):
    n = _log_int(rng, lo, hi)
    pitch = rng.choice([2, 4, 4, 8]) if n <= 1024 else rng.choice([2, 4])
    room = (n * pitch / 4096.0) ** 2 * 200.0  # the benchmark's density
    return {"scene": "polys", "n": n, "pitch": pitch, "polys": max(4, int(min(room, 300) * rng.uniform(0.4, 1.1))),
            "points": rng.randint(1, 5), "segs": rng.randint(0, 2)}


def _draw_maze(rng, most):
    cells = _log_int(rng, 8, most)
    cell = rng.choice([256, 256, 200, 184])
    return {"scene": "maze", "cells": cells, "cell": cell, "n": cells * cell // rng.choice([4, 4, 8]),
            "points": rng.randint(1, 6)}


def draw(rng):
    kind = rng.choice(["map", "map", "map", "map", "host", "frame", "grad", "batch", "paths"])
    if kind == "batch":
        return {"kind": kind, "each": _log_int(rng, 1, 14), "poly_lo": 10, "poly_hi": rng.randint(40, 300)}
    if kind == "grad":
        return dict(_draw_polys(rng, 256, 2048), kind=kind, agents=_log_int(rng, 1000, 100000),
                    tuning="diff2048_grad")
    if kind == "frame":
        return dict(_draw_maze(rng, 40), kind=kind, agents=_log_int(rng, 1000, 100000), tuning="maze2048")
    if kind == "paths":
        return dict(_draw_polys(rng, 256, 1536), kind=kind, queries=rng.randint(8, 48), tuning="polys1024")
    what = rng.choice(["rects", "squares", "polys", "polys", "maze"])
    if what == "rects":
        n = _log_int(rng, 100, 600)
        return {"kind": kind, "scene": what, "n": n, "polys": rng.randint(4, 16), "points": rng.randint(1, 4),
                "segs": 0, "tuning": rng.choice(["rects256", ""])}
    if what == "squares":
        k = rng.choice([2, 4, 6, 8, 10, 14, 20])
        return {"kind": kind, "scene": what, "n": _log_int(rng, 400, 2000) // k * k, "k": k,
                "tuning": rng.choice(["profiling%d" % (k * k), ""])}
    if what == "maze":
        return dict(_draw_maze(rng, 60), kind=kind, tuning=rng.choice(["maze4096", "maze2048", ""]))
    c = dict(_draw_polys(rng, 128, 2048), kind=kind)
    return dict(c, tuning=rng.choice(["polys1024", "diff2048_grad", ""] if c["n"] <= 1024 else
                                     ["polys1024", "diff2048_grad"]))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _scene(case, seed):
    what = case["scene"]
    if what == "rects":
        return sg.plain_rects(seed, W=case["n"], N=case["n"], n_rects=case["polys"], n_points=case["points"])
    if what == "squares":
        return sg.profiling_map(case["k"], W=case["n"], N=case["n"], seed=seed)
    if what == "maze":
        return sg.maze(seed, cells=case["cells"], cell=case["cell"], N=case["n"], n_points=case["points"])
    W = case["n"] * case["pitch"]
    if case["kind"] == "grad":  # movable sources at arbitrary float positions
        return sg.differentiable(seed, W=W, N=case["n"], n_polys=case["polys"], n_points=case["points"],
                                 n_segs=case["segs"], n_agents=case["agents"])
    return sg.tiny(seed, W=W, N=case["n"], n_polys=case["polys"], n_points=case["points"], n_segs=case["segs"],
                   r=(min(20.0, W / 50.0), min(120.0, W / 10.0)), k=(4, 8))


def _moved(case, scene, seed):
    """The frame's sources and agents: every source a few steps from where it was."""
    pts, segs = sg.maze_source_frames(scene, 5, seed=seed)
    r = np.random.RandomState(seed % (1 << 32))
    cells, cell, n = case["cells"], case["cell"], case["agents"]
    c = r.randint(0, cells, (n, 2))
    at = c * cell + r.randint(24, cell - 24, (n, 2))  # in the cells' free interiors
    return pts[4], segs[4], (at * scene.grid[0] // scene.world[0]).astype(np.int32)


def _tuned(scene, key):
    s = spm.Scene(scene)
    if key:
        s.autotune(cache_key=key)
    return s


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        scenes = []
        for k, side in enumerate(SIDES):
            scenes += sg.batched(len(SIDES) * seed + k, n_scenes=case["each"], sides=(side,),
                                 poly_range=(case["poly_lo"], case["poly_hi"]))
        objs = [_tuned(x, "batched256-side%d" % x.grid[0]) for x in scenes]
        n = sum(x.n_pixels for x in scenes)
        dist = torch.empty(n, dtype=torch.float32, device="cuda")
        parent = torch.empty(n, dtype=torch.int32, device="cuda")
        cut = np.cumsum([0] + [x.n_pixels for x in scenes])
        batch = _Batch(objs, [dist[a:b] for a, b in zip(cut[:-1], cut[1:])],
                       [parent[a:b] for a, b in zip(cut[:-1], cut[1:])])
        return {"kind": kind, "batch": batch, "dist": dist, "parent": parent}
    scene = _scene(case, seed)
    s = _tuned(scene, case["tuning"])
    st = {"kind": kind, "scene": s}
    if kind == "grad":
        st["points"] = torch.tensor(scene.points, dtype=torch.float32, device="cuda", requires_grad=True)
        st["segs"] = torch.tensor(scene.segs, dtype=torch.float32, device="cuda", requires_grad=True)
        st["agents"] = torch.tensor(scene.agents, device="cuda")
        return st
    st["dist"], st["parent"] = s.empty_outputs()
    if kind == "host":
        st["dist"], st["parent"] = (torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
                                    for t in (st["dist"], st["parent"]))
    if kind == "frame":
        pts, segs, agents = _moved(case, scene, seed)
        st["points"], st["segs"] = torch.tensor(pts, device="cuda"), torch.tensor(segs, device="cuda")
        st["agents"] = torch.tensor(agents, device="cuda")
        st["loss"] = torch.empty((), dtype=torch.float32, device="cuda")
    if kind == "paths":
        s.compute(st["dist"], st["parent"])
        s.sync()
        st["at"] = _query_points(case, scene, seed)
    return st


class _Batch:
    """A batch that writes into given planes; keeps its scenes alive."""

    def __init__(self, scenes, dist, parent):
        self.scenes = scenes
        self.handle = spm.spm_batch_create([s.handle for s in scenes], dist, parent)

    def __del__(self):
        spm.spm_batch_destroy(self.handle)


def _query_points(case, scene, seed):
    """Free points spread over the world."""
    r = np.random.RandomState((seed + 7) % (1 << 32))
    out = []
    while len(out) < case["queries"]:
        x, y = (float(np.float32(v)) for v in r.uniform(1, scene.world[0] - 1, 2))
        if all(_outside(p, x, y) for p in scene.polys):
            out.append((x, y))
    return out


def _outside(poly, x, y):
    a = poly.astype(np.float64)
    b = np.roll(a, -1, axis=0)
    turn = (b[:, 0] - a[:, 0]) * (y - a[:, 1]) - (b[:, 1] - a[:, 1]) * (x - a[:, 0])
    return turn.min() < -8.0 * np.abs(b - a).max()  # clear of the edge by some units


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(st):
    kind = st["kind"]
    if kind == "batch":
        spm.spm_batch_compute(st["batch"].handle)
        return {"dist": st["dist"], "parent": st["parent"]}
    s = st["scene"]
    if kind == "map":
        s.compute(st["dist"], st["parent"])
    elif kind == "host":
        spm.spm_compute_host(s.handle, None, st["dist"], st["parent"])
    elif kind == "frame":
        s.update_sources_device(st["points"], st["segs"])
        s.compute(st["dist"], st["parent"])
        spm.spm_agents_forward(s.handle, None, st["agents"], st["dist"], st["parent"], st["loss"])
        return {"dist": st["dist"], "parent": st["parent"], "loss": st["loss"]}
    elif kind == "grad":
        loss = spm.agent_loss(s, st["points"], st["segs"], st["agents"])
        gp, gs = torch.autograd.grad(loss, (st["points"], st["segs"]))
        return {"loss": loss, "grad_points": gp, "grad_segs": gs}
    elif kind == "paths":
        paths = np.zeros((len(st["at"]), PATH_CAP, 2), np.float32)
        for k, (x, y) in enumerate(st["at"]):
            p = s.extract_path(x, y, cap=PATH_CAP)
            paths[k, :len(p)] = p
        return {"paths": paths}
    return {"dist": st["dist"], "parent": st["parent"]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    """Every pixel's distance and parent written once, the scene (vertices and
    sources) and the agents read once; 7 operations for a pixel's winning
    distance (two differences, their squares' sum, root, cost)."""
    kind = case["kind"]
    if kind == "batch":
        px = float(case["each"] * sum(n * n for n in SIDES))
        verts = case["each"] * len(SIDES) * 0.5 * (case["poly_lo"] + case["poly_hi"]) * 5.5
        return {"bytes": 8.0 * px + 8.0 * verts, "flops": 7.0 * px}
    if kind == "paths":  # per query its pixel and a short chain of (position, parent) entries
        return {"bytes": case["queries"] * (8.0 + 8 * 12.0), "flops": 10.0 * case["queries"]}
    px = float(case["n"]) ** 2
    if case["scene"] == "maze":
        verts = 4.0 * case["cells"] ** 2 * 1.03
    elif case["scene"] == "squares":
        verts = 4.0 * case["k"] ** 2
    else:
        verts = 5.5 * case["polys"]
    agents = case.get("agents", 0)
    return {"bytes": 8.0 * px + 8.0 * verts + 12.0 * agents, "flops": 7.0 * px + 2.0 * agents}


# ---------------------------------------------------------------------------
# the same outputs in 64 bits
# ---------------------------------------------------------------------------

class _Exact:
    """Geodesic distances among plain convex obstacles in 64 bits: sources and
    polygon vertices are nodes, a link is free when its open segment meets no
    polygon's open interior, node costs are shortest paths over the free
    links, and a point takes the least cost + distance over the nodes it
    sees. Segment sources also count by their perpendicular foot."""

    def __init__(self, polys, points, segs):
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        m = max([len(p) for p in polys] + [3])
        ccw = []
        for p in polys:
            p = np.asarray(p, np.float64)
            q = np.roll(p, -1, axis=0)
            ccw.append(p if (p[:, 0] * q[:, 1] - p[:, 1] * q[:, 0]).sum() > 0 else p[::-1])
        pad = [np.concatenate([p, np.repeat(p[-1:], m - len(p), axis=0)]) for p in ccw]
        self.V = torch.tensor(np.array(pad).reshape(-1, m, 2), dtype=torch.float64, device=self.dev)
        self.E = torch.roll(self.V, -1, 1) - self.V
        self.flat = (self.E == 0).all(-1)  # padding, no edge
        t = lambda v, k: torch.tensor(np.asarray(v, np.float64).reshape(-1, k), device=self.dev)  # noqa: E731
        self.points, self.segs = t(points, 2), t(segs, 4)
        verts = t(np.concatenate(ccw) if ccw else [], 2)
        verts = verts[self.free(verts)]
        self.nodes = torch.cat([self.points, self.segs.reshape(-1, 2), verts])
        self.n_src = len(self.nodes) - len(verts)
        self._costs()

    def free(self, P):
        out = torch.ones(len(P), dtype=torch.bool, device=self.dev)
        for i, part in self._parts(P):
            o = self._turn(part)
            out[i:i + len(part)] = ~((o > 0) | self.flat).all(-1).any(-1) if len(self.V) else True
        return out

    def _parts(self, P):
        step = max(1, int(2e7) // max(1, self.V.shape[0] * self.V.shape[1]))
        return ((i, P[i:i + step]) for i in range(0, len(P), step))

    def _turn(self, P):
        d = P[:, None, None, :] - self.V
        return self.E[..., 0] * d[..., 1] - self.E[..., 1] * d[..., 0]

    def sees(self, P, Q):
        """Which open segments P[i] -> Q[i] (Q: one point or as many) meet no open interior."""
        if not len(self.V):
            return torch.ones(len(P), dtype=torch.bool, device=self.dev)
        Q = Q.expand(len(P), 2)
        out = torch.ones(len(P), dtype=torch.bool, device=self.dev)
        for i, p in self._parts(P):
            q = Q[i:i + len(p)]
            inner = ((self._turn(p) > 0) | (self._turn(q) > 0) | self.flat).all(-1)
            d, w = (q - p)[:, None, None, :], self.V - p[:, None, None, :]
            s = d[..., 0] * w[..., 1] - d[..., 1] * w[..., 0]
            out[i:i + len(p)] = ~(inner & (s > 0).any(-1) & (s < 0).any(-1)).any(-1)
        return out

    def feet(self, P):
        """(distance or inf, foot's place on the segment) of every point to every segment's open interior."""
        for k in range(len(self.segs)):
            a, b = self.segs[k, :2], self.segs[k, 2:]
            t = ((P - a) @ (b - a)) / ((b - a) @ (b - a))
            foot = a + t[:, None] * (b - a)
            d = (P - foot).norm(dim=1)
            ok = (t > 0) & (t < 1)
            ok[ok.clone()] = self.sees(P[ok], foot[ok])
            yield k, torch.where(ok, d, math.inf), t

    def _costs(self):
        n, ns = len(self.nodes), self.n_src
        self.cost = torch.full((n,), math.inf, dtype=torch.float64, device=self.dev)
        self.par = torch.full((n,), -1, dtype=torch.int64, device=self.dev)
        self.cost[:ns] = 0
        for k, d, _ in self.feet(self.nodes):
            better = d < self.cost
            self.cost = torch.where(better, d, self.cost)
            self.par[better] = -2 - k  # from segment k's interior
        L = torch.cdist(self.nodes, self.nodes, compute_mode="donot_use_mm_for_euclid_dist")
        for u in range(n):
            L[u, ~self.sees(self.nodes, self.nodes[u])] = math.inf
        for _ in range(n):
            best, u = (self.cost[:, None] + L).min(0)
            better = best < self.cost
            better[:ns] = False
            if not better.any():
                break
            self.cost = torch.where(better, best, self.cost)
            self.par = torch.where(better, u, self.par)

    def field(self, P):
        """(distance, node, or -2 - k for segment k's interior, or -1) of every point."""
        best = torch.full((len(P),), math.inf, dtype=torch.float64, device=self.dev)
        par = torch.full((len(P),), -1, dtype=torch.int64, device=self.dev)
        ok = self.free(P)
        for k, d, _ in self.feet(P):
            better = ok & (d < best)
            best[better], par[better] = d[better], -2 - k
        for u in torch.argsort(self.cost, stable=True).tolist():
            if not math.isfinite(float(self.cost[u])):
                break
            d = self.cost[u] + (P - self.nodes[u]).norm(dim=1)
            at = (ok & (d < best)).nonzero()[:, 0]
            if len(at):
                at = at[self.sees(P[at], self.nodes[u])]
                best[at], par[at] = d[at], u
        return best, par


def _centres(scene, at=None):
    (nx, ny), (wx, wy) = scene.grid, scene.world
    if at is None:
        j, i = np.divmod(np.arange(nx * ny), nx)
    else:
        i, j = at[:, 0], at[:, 1]
    return np.stack([(i + 0.5) * (wx / nx), (j + 0.5) * (wy / ny)], 1)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "paths"):  # millions of pixels; and which of a pixel's points a path
        return None                 # takes first depends on the grid
    if kind == "grad":
        return _exact_grad(case, seed)
    verts = {"maze": 4 * case.get("cells", 0) ** 2, "squares": 4 * case.get("k", 0) ** 2}.get(
        case["scene"], 5 * case.get("polys", 0))
    if float(case["n"]) ** 2 * verts ** 2 > 8e10:
        return None  # over 20 seconds of visibility tests
    scene = _scene(case, seed)
    points, segs = scene.points, scene.segs
    agents = None
    if kind == "frame":
        points, segs, agents = _moved(case, scene, seed)
    e = _Exact(scene.polys, points, segs)
    P = torch.tensor(_centres(scene), device=e.dev)
    dist = e.field(P)[0].reshape(scene.grid[1], scene.grid[0])
    if kind != "frame":
        return {"dist": dist, "parent": None}
    at = torch.tensor(agents, dtype=torch.int64, device=e.dev)
    d = dist[at[:, 1], at[:, 0]]
    return {"dist": dist, "parent": None, "loss": torch.where(torch.isfinite(d), d, 0.0).mean()}


def _exact_grad(case, seed):
    scene = _scene(case, seed)
    if len(scene.agents) * (5.0 * case["polys"]) ** 2 > 8e10:
        return None
    e = _Exact(scene.polys, np.float32(scene.points), np.float32(scene.segs))
    at, back = np.unique(scene.agents, axis=0, return_inverse=True)
    P = torch.tensor(_centres(scene, at), device=e.dev)
    _, par = e.field(P)
    # the root link of every agent: the last point before its source
    x, node, rest = P.clone(), par.clone(), torch.zeros(len(P), dtype=torch.float64, device=e.dev)
    while True:
        inner = node >= e.n_src
        if not inner.any():
            break
        u = node[inner]
        rest[inner] += (x[inner] - e.nodes[u]).norm(dim=1)
        x[inner], node[inner] = e.nodes[u], e.par[u]
    points = e.points.clone().requires_grad_()
    segs = e.segs.clone().requires_grad_()
    src = torch.cat([points, segs.reshape(-1, 2)])
    d = rest.clone()
    at_node = node >= 0
    d = d + torch.where(at_node, (x - src[node.clamp(min=0)]).norm(dim=1), torch.zeros_like(d))
    if len(segs):
        k = (-2 - node).clamp(min=0)
        a, b = segs[k, :2], segs[k, 2:]
        v = b - a
        off = (v[:, 0] * (x - a)[:, 1] - v[:, 1] * (x - a)[:, 0]).abs() / v.norm(dim=1)
        d = d + torch.where(node <= -2, off, torch.zeros_like(d))
    loss = d[torch.tensor(back.reshape(-1), device=e.dev)].mean()
    gp, gs = torch.autograd.grad(loss, (points, segs), allow_unused=True)
    zero = lambda g, v: torch.zeros_like(v) if g is None else g  # noqa: E731
    return {"loss": loss.detach(), "grad_points": zero(gp, points), "grad_segs": zero(gs, segs)}
