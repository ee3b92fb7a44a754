"""The work a user has this library do, as timed cases.

Each case is one call (or one short sequence of calls) of the public Python
entry points on seeded synthetic triangulations.  Meshes are made on the GPU:

* grids: jittered rows x cols vertices on the unit square (+-0.3 of a cell),
  a random diagonal per cell, row-major order -- the recipe of
  ``meshgen.perturbed_grid`` (every vertex of the exact-grid paper generator
  moved a little);
* random meshes: ``meshgen.random_delaunay`` itself (uniform points, convex
  hull and its slivers, made on the host, so not for the largest sizes);
* Delaunay meshes: the same kind of mesh made on the GPU on the unit square:
  scattered points (the grid's vertices moved by several random steps of half
  a cell), brought to the Delaunay triangulation by edge flips, vertices
  numbered along a Hilbert curve and triangles sorted by their vertices, the
  order ``meshgen.random_delaunay`` gives.

A batch or a request stream mixes both alternately, sizes log-uniform, as
``meshgen.random_batch`` does.  All outputs are whole numbers.
"""
from __future__ import annotations

import json
import math
import zlib

import numpy as np
import torch

from paper_2403_14723_gb300 import meshgen, polylla


# ---------------------------------------------------------------------------
# mesh generation (torch, on the GPU)
# ---------------------------------------------------------------------------

def _hilbert(xy: torch.Tensor) -> torch.Tensor:
    """Hilbert curve index of points of the unit square (16 bits a side)."""
    n = 1 << 16
    q = (xy * n).long().clamp_(0, n - 1)
    x, y = q[:, 0].clone(), q[:, 1].clone()
    d = torch.zeros_like(x)
    s = n >> 1
    while s:
        rx, ry = (x & s) > 0, (y & s) > 0
        d += s * s * ((3 * rx.long()) ^ ry.long())
        turn, rot = ~ry & rx, ~ry
        x, y = torch.where(turn, n - 1 - x, x), torch.where(turn, n - 1 - y, y)
        x, y = torch.where(rot, y, x), torch.where(rot, x, y)
        s >>= 1
    return d


def _area2(xy, a, b, c):
    p, q, r = xy[a], xy[b], xy[c]
    return (q[:, 0] - p[:, 0]) * (r[:, 1] - p[:, 1]) - (q[:, 1] - p[:, 1]) * (r[:, 0] - p[:, 0])


def _next3(e):
    return e - e % 3 + (e + 1) % 3


def _flip_to_delaunay(xy, org, twin, movable, most: int = 80):
    """Edge flips until no edge of a triangle with ``movable`` is non-Delaunay.
    Every round flips a set of edges that share no triangle."""
    e = torch.arange(org.numel(), device=org.device)
    mine = movable[e // 3]                           # slots keep their mesh: flips move edges inside it
    triangles = org.numel() // 3
    for k in range(most):
        cand = e[(twin > e) & mine]
        f = twin[cand]
        ia, ib = org[cand], org[f]
        ic, idd = org[_next3(_next3(cand))], org[_next3(_next3(f))]
        d = xy[idd]
        ax, ay = (xy[ia] - d).unbind(1)
        bx, by = (xy[ib] - d).unbind(1)
        cx, cy = (xy[ic] - d).unbind(1)
        a2, b2, c2 = ax * ax + ay * ay, bx * bx + by * by, cx * cx + cy * cy
        det = a2 * (bx * cy - cx * by) - b2 * (ax * cy - cx * ay) + c2 * (ax * by - bx * ay)
        bad = det > 1e-10 * (a2 + b2 + c2) ** 2
        bad &= (_area2(xy, ic, idd, ib) > 0) & (_area2(xy, idd, ic, ia) > 0)
        cand, f = cand[bad], f[bad]
        if cand.numel() == 0:
            break
        key = (cand * 0x9E3779B1 + 0x7F4A7C15 * (k + 1)) & 0x7FFFFFFF
        key = key * (1 << 32) + cand
        low = torch.full((triangles,), torch.iinfo(torch.int64).max, device=org.device)
        low.scatter_reduce_(0, cand // 3, key, "amin")
        low.scatter_reduce_(0, f // 3, key, "amin")
        go = (low[cand // 3] == key) & (low[f // 3] == key)
        x, y = cand[go], f[go]
        xn, yn = _next3(x), _next3(y)
        xp, yp = _next3(xn), _next3(yn)
        a, b, c, d = org[x], org[y], org[xp], org[yp]
        # the triangles (c d b) and (d c a) take the places of (a b c) and (b a d)
        place = e.clone()
        place[yp], place[xn], place[xp], place[yn] = xn, xp, yn, yp
        moved = torch.where(twin >= 0, place[twin.clamp_min(0)], twin)
        twin = torch.empty_like(twin)
        twin[place] = moved
        twin[x], twin[y] = y, x
        org = org.clone()
        org[x], org[xn], org[xp] = c, d, b
        org[y], org[yn], org[yp] = d, c, a
    return org, twin


def _scatter_points(xy, org, twin, fixed, movable, cell, gen, steps: int = 8):
    """Random steps of the inner points, each kept only where every triangle
    stays counter-clockwise, with flips between them."""
    tri = org.view(-1, 3)
    for _ in range(steps):
        step = (torch.rand(xy.shape, generator=gen, device=xy.device, dtype=torch.float64) - 0.5) * 1.2 * cell
        step[fixed] = 0
        for _ in range(60):
            new = xy + step
            bad = _area2(new, tri[:, 0], tri[:, 1], tri[:, 2]) <= 0
            if not bool(bad.any()):
                break
            step[tri[bad].reshape(-1)] = 0
        else:
            continue
        xy = new
        org, twin = _flip_to_delaunay(xy, org, twin, movable)
        tri = org.view(-1, 3)
    return xy, org, twin


def _triangulations(shapes, kinds, seed: int, device):
    """Triangulations of ``shapes`` [(rows, cols)] vertices, each ``kinds[i]``
    "grid" or "delaunay", one after the other: coordinates, the vertex each
    half-edge leaves, its twin (-1: on the border), and the vertex and
    triangle prefix sums."""
    gen = torch.Generator(device=device)
    gen.manual_seed(seed)
    dev = {"device": device}
    R = torch.tensor([r for r, _ in shapes], **dev)
    C = torch.tensor([c for _, c in shapes], **dev)
    V, Q = R * C, (R - 1) * (C - 1)
    n = len(shapes)
    voff = torch.zeros(n + 1, dtype=torch.int64, **dev)
    voff[1:] = V.cumsum(0)
    toff = torch.zeros(n + 1, dtype=torch.int64, **dev)
    toff[1:] = 2 * Q.cumsum(0)
    # vertices
    vm = torch.repeat_interleave(torch.arange(n, **dev), V)
    lv = torch.arange(vm.numel(), **dev) - voff[vm]
    i, j = lv // C[vm], lv % C[vm]
    cell = torch.stack([1.0 / (C[vm] - 1).double(), 1.0 / (R[vm] - 1).double()], 1)
    xy = torch.stack([j.double(), i.double()], 1) * cell
    fixed = (i == 0) | (i == R[vm] - 1) | (j == 0) | (j == C[vm] - 1)
    jit = (torch.rand(xy.shape, generator=gen, dtype=torch.float64, **dev) - 0.5) * 0.6 * cell
    jit[fixed] = 0
    xy = (xy + jit).clamp_(0, 1)
    # cells and their triangles, by the diagonal of a coin (the other one
    # where that would leave a triangle without area)
    cm = torch.repeat_interleave(torch.arange(n, **dev), Q)
    lc = torch.arange(cm.numel(), **dev) - toff[cm] // 2
    w = C[cm] - 1
    p = voff[cm] + (lc // w) * C[cm] + lc % w
    s = C[cm]
    coin = torch.randint(0, 2, (cm.numel(),), generator=gen, **dev).bool()
    okA = (_area2(xy, p, p + 1, p + s + 1) > 0) & (_area2(xy, p, p + s + 1, p + s) > 0)
    okB = (_area2(xy, p, p + 1, p + s) > 0) & (_area2(xy, p + 1, p + s + 1, p + s) > 0)
    A = torch.where(coin, okA, ~okB)
    tri = torch.empty((cm.numel(), 2, 3), dtype=torch.int64, **dev)
    tri[:, 0, 0], tri[:, 0, 1] = p, p + 1
    tri[:, 0, 2] = torch.where(A, p + s + 1, p + s)
    tri[:, 1, 0] = torch.where(A, p, p + 1)
    tri[:, 1, 1], tri[:, 1, 2] = p + s + 1, p + s
    del lc, w, coin, okA, okB, A
    org = tri.reshape(-1)
    T = org.numel() // 3
    # twins from the closed-form edge numbers (smaller vertex, direction)
    e = torch.arange(3 * T, **dev)
    dst = org[_next3(e)]
    lo = torch.minimum(org, dst)
    step, col = torch.maximum(org, dst) - lo, C[vm[org]]
    kind = torch.where(step == 1, 0, torch.where(step == col, 1, torch.where(step == col + 1, 2, 3)))
    # with two columns the steps 1 and col - 1 are the same number: the
    # column tells them apart
    kind = torch.where((step == 1) & (col == 2) & (lv[lo] % 2 == 1), 3, kind)
    eid = 4 * lo + kind
    del step, col, kind, lo
    up = org < dst
    half = torch.full((2, 4 * vm.numel()), -1, dtype=torch.int64, **dev)
    half[0, eid[up]] = e[up]
    half[1, eid[~up]] = e[~up]
    twin = torch.where(up, half[1, eid], half[0, eid])
    del half, eid, up, dst
    dl = torch.tensor([k == "delaunay" for k in kinds], **dev)
    tm = torch.repeat_interleave(torch.arange(n, **dev), 2 * Q)
    if bool(dl.any()):
        still = fixed | ~dl[vm]
        org, twin = _flip_to_delaunay(xy, org, twin, dl[tm])
        xy, org, twin = _scatter_points(xy, org, twin, still, dl[tm], cell, gen)
        # vertices along a Hilbert curve, triangles by their vertex ids
        # (grids keep their order)
        key = torch.where(dl[vm], _hilbert(xy), lv)
        order = torch.argsort(vm * (1 << 33) + key, stable=True)
        rank = torch.empty_like(order)
        rank[order] = torch.arange(order.numel(), **dev)
        xy, org = xy[order], rank[org]
        tri = org.view(-1, 3)
        first = torch.where(dl[tm], tri.argmin(1), 0)
        turn = (first[:, None] + torch.arange(3, **dev)) % 3
        tri = tri.gather(1, turn)
        key = torch.where(dl[tm], tri[:, 0] * vm.numel() + tri[:, 1],
                          (voff[tm] * vm.numel()) + torch.arange(T, **dev) - toff[tm])
        order = torch.argsort(key, stable=True)
        old = (3 * torch.arange(T, **dev)[:, None] + turn)[order].reshape(-1)   # new slot -> old slot
        place = torch.empty_like(old)
        place[old] = e
        org = tri[order].reshape(-1)
        tw = twin[old]
        twin = torch.where(tw >= 0, place[tw.clamp_min(0)], tw)
        del key, order, old, place, tw, turn, tri
    return xy, org, twin, voff, toff


def _random(points: int, seed: int, device):
    """``meshgen.random_delaunay`` in the form of :func:`_triangulations`."""
    m = meshgen.random_delaunay(points, seed=seed)
    T = m.n_triangles
    twin = np.where(m.twin[:3 * T] < 3 * T, m.twin[:3 * T], -1)
    put = [torch.from_numpy(np.ascontiguousarray(a)).to(device) for a in (m.coords, m.origin[:3 * T].astype(np.int64),
                                                                        twin.astype(np.int64))]
    return (*put, torch.tensor([0, m.n_vertices], device=device), torch.tensor([0, T], device=device))


def make_meshes(shapes, kinds, shape_seed: int, seed: int, device="cuda") -> dict:
    """Meshes in the library's half-edge layout, concatenated with local
    indices: coords, origin, twin, next, prev and the host prefix sums.
    ``shape_seed`` draws the triangulations; ``seed`` says how each is
    numbered (where on its curve or row the vertices and the triangles start)
    and placed (quarter turns, a scale by a power of two: both exact), so that
    the meshes of two seeds have no array in common and the same number of
    triangles and polygons."""
    dev = {"device": device}
    n = len(shapes)
    if kinds == ["random"]:
        xy, org, twin, voff, toff = _random(shapes[0], shape_seed, device)
    else:
        xy, org, twin, voff, toff = _triangulations(shapes, kinds, shape_seed, device)
    V, T = voff[1:] - voff[:-1], int(toff[-1])
    vm = torch.repeat_interleave(torch.arange(n, **dev), V)
    tm = torch.repeat_interleave(torch.arange(n, **dev), toff[1:] - toff[:-1])
    rng = np.random.default_rng(int(seed) % (1 << 62))
    vshift, tshift, quarter = (torch.from_numpy(rng.integers(0, 1 << 30, size=n)).to(device) for _ in range(3))
    scale = torch.from_numpy(2.0 ** rng.integers(-3, 4, size=n)).to(device)
    for k in range(4):
        turned = torch.stack([-xy[:, 1], xy[:, 0]], 1) if k else xy
        xy = torch.where((quarter % 4 >= k)[vm][:, None], turned, xy)
    xy = xy * scale[vm][:, None]
    rank = voff[vm] + (torch.arange(vm.numel(), **dev) - voff[vm] + vshift[vm]) % V[vm]
    moved = torch.empty_like(xy)
    moved[rank] = xy
    xy, org = moved, rank[org]
    rank = toff[tm] + (torch.arange(T, **dev) - toff[tm] + tshift[tm]) % (toff[1:] - toff[:-1])[tm]
    e = torch.arange(3 * T, **dev)
    place = 3 * rank.repeat_interleave(3) + e % 3
    o, w = torch.empty_like(org), torch.empty_like(twin)
    o[place] = org
    w[place] = torch.where(twin >= 0, place[twin.clamp_min(0)], twin)
    org, twin = o, w
    del o, w, place, rank, moved
    # border half-edges, one per boundary edge
    src = e[twin < 0]
    bm = tm[src // 3]
    nb = torch.bincount(bm, minlength=n)
    boff = torch.zeros(n + 1, dtype=torch.int64, **dev)
    boff[1:] = nb.cumsum(0)
    hoff = 3 * toff + boff
    rank = torch.arange(src.numel(), **dev)
    borg, bdst = org[_next3(src)], org[src]
    out_of = torch.empty(vm.numel(), dtype=torch.int64, **dev)
    out_of[borg] = rank
    bnext = out_of[bdst]
    bprev = torch.empty_like(bnext)
    bprev[bnext] = rank
    b0 = 3 * (toff[1:] - toff[:-1])[bm] - boff[bm]                   # border rank -> local half-edge
    t3 = 3 * toff[tm].repeat_interleave(3)
    at = e - t3 + hoff[tm].repeat_interleave(3)                      # interior slot -> place in the arrays
    bat = hoff[bm] + b0 + rank
    H = int(hoff[-1])
    out = {k: torch.empty(H, dtype=torch.int32, **dev) for k in ("origin", "twin", "next", "prev")}
    ltwin = twin - t3
    ltwin[src] = b0 + rank
    out["origin"][at] = (org - voff[tm].repeat_interleave(3)).int()
    out["twin"][at] = ltwin.int()
    out["next"][at] = (_next3(e) - t3).int()
    out["prev"][at] = (_next3(_next3(e)) - t3).int()
    out["origin"][bat] = (borg - voff[bm]).int()
    out["twin"][bat] = (src - 3 * toff[bm]).int()
    out["next"][bat] = (b0 + bnext).int()
    out["prev"][bat] = (b0 + bprev).int()
    out["coords"] = xy.contiguous()
    for k, v in (("vertex_offset", voff), ("triangle_offset", toff), ("halfedge_offset", hoff)):
        out[k] = v.cpu().numpy().astype(np.int32)
    return out


def _shape_seed(case) -> int:
    """A seed of the case's own values."""
    return zlib.crc32(json.dumps({k: v for k, v in case.items() if k != "name"}, sort_keys=True).encode())


def _meshes(case, seed, device="cuda"):
    if "meshes" in case:
        shapes, kinds = _mix(case)
    elif case["mesh"] == "random":
        shapes, kinds = [case["points"]], ["random"]
    else:
        shapes, kinds = [(case["rows"], case["cols"])], [case["mesh"]]
    return make_meshes(shapes, kinds, _shape_seed(case), seed, device)


def _host_meshes(m):
    a = {k: m[k].cpu().numpy() for k in ("coords", "origin", "twin", "next", "prev")}
    vo, to, ho = m["vertex_offset"], m["triangle_offset"], m["halfedge_offset"]
    return [meshgen.HalfEdgeMesh(coords=a["coords"][vo[i]:vo[i + 1]],
                                 **{k: a[k][ho[i]:ho[i + 1]] for k in ("origin", "twin", "next", "prev")},
                                 n_triangles=int(to[i + 1] - to[i])) for i in range(len(to) - 1)]


def _side(t: float) -> int:
    return max(2, int(round(math.sqrt(t / 2.0))) + 1)


def _mix(case):
    """Shapes and kinds of a batch: log-uniform sizes, alternately Delaunay
    and grids; the sizes come from the case alone."""
    rng = np.random.default_rng(int(case["sizes"]))
    t = np.exp(rng.uniform(math.log(case["t_min"]), math.log(case["t_max"]), size=case["meshes"]))
    shapes = []
    for v in t:
        s = _side(v)
        shapes.append((s, max(2, s + int(rng.integers(-(s // 4), s // 4 + 1)))))
    return shapes, ["delaunay" if i % 2 == 0 else "grid" for i in range(case["meshes"])]


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the smallest meshes of a batch, meshed one at a time: the latency of a call
        {"name": "delaunay_100", "call": "generate", "mesh": "random", "points": 52},
        # the paper's small random set (2,000 points)
        {"name": "delaunay_2k", "call": "generate", "mesh": "random", "points": 2000},
        # an ordinary grid with odd sides (the 300-vertex grid of the parity tests, made ragged)
        {"name": "grid_301", "call": "generate", "mesh": "grid", "rows": 301, "cols": 297},
        # an ordinary random mesh (400 k triangles), long polygons along its hull among the rest
        {"name": "delaunay_200k", "call": "generate", "mesh": "random", "points": 200_003},
        # as many triangles as the paper's 1 M random points give
        {"name": "delaunay_1m", "call": "generate", "mesh": "delaunay", "rows": 1000, "cols": 1000},
        # the headline mesh: 33.5 M triangles
        {"name": "grid_4096", "call": "generate", "mesh": "grid", "rows": 4096, "cols": 4096},
        # a caller that may not allocate, close to that entry point's limit
        {"name": "noalloc_130k", "call": "noalloc", "mesh": "random", "points": 65_001},
        # many meshes at once: 100 to 200,000 triangles each, Delaunay and grids
        {"name": "batch_512", "call": "batch", "meshes": 512, "t_min": 100, "t_max": 200_000, "sizes": 4},
        # post-processing: convex polygons from a random mesh (1 M triangles)
        {"name": "convex_500k", "call": "convexify", "mesh": "delaunay", "rows": 701, "cols": 713},
        # the Lepp primitive over every triangle of a labelled mesh (8 M triangles)
        {"name": "lepp_grid_2048", "call": "lepp", "mesh": "grid", "rows": 2048, "cols": 2047},
        # a mesh in pinned host memory, copies in and out included (0.5 M triangles)
        {"name": "host_500k", "call": "host", "mesh": "delaunay", "rows": 499, "cols": 503},
        # requests of 1 k to 50 k triangles through the serving loop, all waiting at once
        {"name": "served_16", "call": "served", "meshes": 16, "t_min": 1000, "t_max": 50_000, "sizes": 5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["generate", "generate", "generate", "generate", "noalloc", "batch", "convexify", "lepp", "host",
                       "served"])
    if call in ("batch", "served"):
        n = _log_int(rng, 2, 400) if call == "batch" else rng.randint(1, 24)
        return {"call": call, "meshes": n, "t_min": 100 if call == "batch" else 1000,
                "t_max": _log_int(rng, 5_000, 150_000) if call == "batch" else 50_000,
                "sizes": rng.randrange(1 << 20)}
    mesh = rng.choice(["grid", "delaunay", "random"])
    most = {"noalloc": 125_000, "convexify": 4_000_000, "lepp": 16_000_000, "host": 2_000_000}.get(call, 30_000_000)
    if mesh == "random":
        return {"call": call, "mesh": mesh, "points": _log_int(rng, 20, min(most, 400_000) / 2)}
    if mesh == "delaunay":
        most = min(most, 4_000_000)
    s = _side(_log_int(rng, 60, most * 0.8))
    return {"call": call, "mesh": mesh, "rows": s, "cols": max(2, int(s * rng.uniform(0.8, 1.25)))}


class _Batch:
    """A batch context and the arrays it works on."""

    def __init__(self, m):
        self.batch = polylla.DeviceBatch(*(m[k] for k in ("coords", "origin", "twin", "next", "prev", "vertex_offset",
                                                          "triangle_offset", "halfedge_offset")))
        self.ctx = polylla.polylla_batch_create(self.batch)

    def __del__(self):
        polylla.polylla_destroy(self.ctx)


class _Host:
    """A host-buffer context and pinned buffers."""

    def __init__(self, mesh):
        r = polylla.HostRequest(mesh)
        self.inp, self.out = r.inp, r.out
        self.ctx = polylla.polylla_create_host(mesh.n_vertices, mesh.n_triangles, mesh.n_halfedges)

    def __del__(self):
        polylla.polylla_destroy(self.ctx)


class _Served:
    """A server and pinned requests."""

    def __init__(self, meshes):
        self.requests = [polylla.HostRequest(m) for m in meshes]
        self.server = polylla.Server(1 << 30)

    def __del__(self):
        self.server.close()


def prepare(case, seed):
    call = case["call"]
    m = _meshes(case, seed)
    if call == "batch":
        return call, _Batch(m)
    if call == "served":
        return call, _Served(_host_meshes(m))
    if call == "host":
        return call, _Host(_host_meshes(m)[0])
    mesh = polylla.DeviceMesh(m["coords"], m["origin"], m["twin"], m["next"], m["prev"], int(m["triangle_offset"][-1]))
    if call == "noalloc":
        T = mesh.n_triangles
        new = [torch.zeros(k, dtype=torch.int32, device="cuda") for k in (T, T + 1, 3 * T, 3 * T, 3)]
        return call, (mesh, new)
    p = polylla.Polylla(mesh)
    if call == "lepp":
        p.generate()   # the labels the paths follow
    return call, p


def _owned(out, owner):
    """Outputs that live in a context's own memory: they keep it alive."""
    for t in out.values():
        if isinstance(t, torch.Tensor):
            t.owner = owner
    return out


def run(state):
    call, s = state
    if call == "batch":
        polylla.polylla_generate(s.ctx)
        out = polylla.polylla_get_polygons(s.ctx)
        out["poly_offset"] = polylla.polylla_batch_polygon_offsets(s.ctx, s.batch.n_meshes)
        return {**_owned(out, s), "next": s.batch.next, "prev": s.batch.prev}
    if call == "served":
        tickets = [s.server.submit(r) for r in s.requests]
        infos = [s.server.wait(t) for t in tickets]
        every = [r.result(i) for r, i in zip(s.requests, infos)]
        return {k: np.concatenate([r[k] for r in every]) for k in every[0]}
    if call == "host":
        P, NF = polylla.polylla_generate_host(s.ctx, s.inp, s.out)
        n = {"seeds": P, "offsets": P + 1, "he_list": NF, "v_list": NF}
        return {k: t[:n.get(k, t.numel())] for k, t in s.out.items()}
    if call == "noalloc":
        mesh, new = s
        polylla.polylla_generate_noalloc(mesh, *new)
        return [*new, mesh.next, mesh.prev]
    if call == "lepp":
        return polylla.polylla_lepp_terminal(s.ctx, s.mesh.n_triangles)
    s.generate()
    if call == "convexify":
        s.convexify()
    return {**_owned(s.polygons(), s), "next": s.mesh.next, "prev": s.mesh.prev}


# polygons per triangle, as they come out on such meshes; a polygon of k
# triangles has k + 2 half-edges, so N_F = T + 2 P
_POLYGONS = {"grid": 0.392, "delaunay": 0.17, "random": 0.16}


def work(case):
    """Bytes: coords, origin and twin in, next and prev of the interior
    half-edges and the polygon lists out (Lepp: twin in, two words a triangle
    out; host calls: the same bytes, once over the link)."""
    if "meshes" in case:
        shapes, kinds = _mix(case)
    elif case["mesh"] == "random":   # 2 n - 2 - hull triangles
        shapes, kinds = [(2, case["points"])], ["random"]
    else:
        shapes, kinds = [(case["rows"], case["cols"])], [case["mesh"]]
    total = flops = 0.0
    for (r, c), k in zip(shapes, kinds):
        V, T = r * c, 2 * (r - 1) * (c - 1)
        V = c if k == "random" else V
        if case["call"] == "lepp":
            total += 12 * T + 8 * T
            continue
        P = _POLYGONS[k] * T * (1.3 if case["call"] == "convexify" else 1.0)
        total += 16 * V + 24 * T + 24 * T + 8 * (T + 2 * P) + 8 * P
        flops += 15 * T    # the squared lengths
    return {"bytes": total, "flops": flops}
