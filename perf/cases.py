"""The calls that a user of the engine makes, with sizes, inputs and outputs, for timing and comparing.

`listed()` names the standing cases, `draw()` gives further ones of the same ranges, `prepare()` builds a
case's graph handle and buffers on the GPU from a seed, `run()` makes one pass through the public entry
points, `work()` counts what a pass cannot do without, and `exact()` gives the answer in 64 bits by plain
torch.  The graph families and sizes are those of this repository's workloads: 4-neighbour grids, the
road-shaped grid, R-MAT, G(n, m) and random directed graphs.
"""
from __future__ import annotations

import math

import torch

import paper_2602_10080_gb300 as S

INF = 0xFFFFFFFF


def listed():
    return [
        # the smallest call: a routing question on a small directed network, where launches and
        # latency are all there is
        {"name": "directed_1k_pred", "call": "solve", "family": "directed", "n": 1000, "m": 6000, "hi": 100,
         "wtype": "u32", "pred": True},
        # a small map or mesh, with the routes
        {"name": "grid256_pred", "call": "solve", "family": "grid", "W": 256, "H": 256, "hi": 100,
         "wtype": "u32", "pred": True},
        # a mesh of a million vertices, distances only: high diameter, a thin wavefront
        {"name": "grid1024", "call": "solve", "family": "grid", "W": 1024, "H": 1024, "hi": 100,
         "wtype": "u32", "pred": False},
        # a country-sized road network with the routes: 16.8M vertices, 64M arcs
        {"name": "road4096_pred", "call": "solve", "family": "road", "W": 4096, "H": 4096, "hi": 1000,
         "wtype": "u32", "pred": True},
        # the headline: a power-law graph of 134M arcs with predecessors
        {"name": "rmat22_pred", "call": "solve", "family": "rmat", "scale": 22, "ef": 16, "hi": 255,
         "wtype": "u32", "pred": True},
        # real-valued lengths on a graph without hubs, distances only
        {"name": "er21_f32", "call": "solve", "family": "er", "n": 1 << 21, "m": 1 << 25, "hi": 1,
         "wtype": "f32", "pred": False},
        # hop levels and parents on the power-law graph
        {"name": "bfs_rmat22", "call": "bfs", "family": "rmat", "scale": 22, "ef": 16, "hi": 255,
         "wtype": "u32", "pred": True},
        # many sources at once (distance tables, centrality samples): 256 queries in one call
        {"name": "batch256_rmat20", "call": "batch", "nq": 256, "family": "rmat", "scale": 20, "ef": 16,
         "hi": 255, "wtype": "u32", "pred": False},
        # the same with real-valued lengths and fewer queries
        {"name": "batch64_rmat18_f32", "call": "batch", "nq": 64, "family": "rmat", "scale": 18, "ef": 16,
         "hi": 1, "wtype": "f32", "pred": False},
        # a few routes at once on a ragged mesh, with predecessors
        {"name": "batch13_grid_pred", "call": "batch", "nq": 13, "family": "grid", "W": 301, "H": 257, "hi": 100,
         "wtype": "u32", "pred": True},
        # a burst of queries handed to the server, to the last answer
        {"name": "serve24_rmat18", "call": "serve", "nq": 24, "family": "rmat", "scale": 18, "ef": 16, "hi": 255,
         "wtype": "u32", "pred": False},
        # the caller who may not allocate: the CSR as it is, validated and solved in one call
        {"name": "noalloc_rmat13_pred", "call": "noalloc", "family": "rmat", "scale": 13, "ef": 16, "hi": 255,
         "wtype": "u32", "pred": True},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["solve", "solve", "solve", "solve", "bfs", "batch", "batch", "serve", "noalloc"])
    family = rng.choice(["grid", "rmat", "er", "directed"] + (["road"] if call in ("solve", "bfs") else []))
    wtype = rng.choice(["u32", "u32", "f32"])
    # predecessors where they are unique (whole weights of at least one)
    pred = (wtype == "u32" or call == "bfs") and rng.random() < 0.5
    c = {"call": call, "family": family, "wtype": wtype, "pred": pred}
    nq = _log(rng, 2, 256) if call == "batch" else _log(rng, 4, 48) if call == "serve" else 1
    if nq > 1:
        c["nq"] = nq
    # arcs; the solve without allocation has fixed queues, and is for the smaller graphs
    room = (1 << 28) // nq if nq > 1 else 1 << (18 if call == "noalloc" else 27)
    if family == "grid":
        most = min(1024, math.isqrt(room // 4), 512 if nq > 1 else 1024)
        c.update(W=_log(rng, 24, most), H=_log(rng, 24, most), hi=rng.choice([9, 100, 1000]))
    elif family == "road":
        c.update(W=_log(rng, 200, 4096), H=_log(rng, 200, 4096), wtype="u32", pred=rng.random() < 0.5, hi=1000)
    elif family == "rmat":
        most = 18 if call == "serve" else 21
        ef = rng.randint(6, 16)
        while (2 * ef << most) > room:
            most -= 1
        c.update(scale=rng.randint(10, most), ef=ef, hi=rng.choice([15, 255, 1000]))
    else:
        n = _log(rng, 300, min(1 << (18 if nq > 1 else 21), room // 24))
        deg = rng.randint(3, 12)
        c.update(n=n, m=n * deg + rng.randint(0, n - 1), hi=rng.choice([15, 100, 1000]))
    if c["wtype"] == "f32":
        c["hi"] = 1
    return c


# ---------------------------------------------------------------- inputs

def _csr(n, u, v):
    """Sorted CSR of the distinct arcs (u, v), self-loops dropped."""
    key = torch.unique((u * n + v)[u != v])
    u, v = key // n, key % n
    row = torch.zeros(n + 1, dtype=torch.int64, device=u.device)
    row[1:] = torch.cumsum(torch.bincount(u, minlength=n), 0)
    return row.to(torch.int32), v.to(torch.int32), u


def _weights(u, v, salt, hi, wtype):
    """One weight per unordered pair, a hash of its ends: u32 in [1, hi], f32 in (0, 1]."""
    a, b = torch.minimum(u, v), torch.maximum(u, v)
    h = a * 0x9E3779B97F4A7C1 + b * 0x632BE59BD9B4E01 + (salt * 0x3C6EF372FE94F82 & (1 << 62) - 1)
    for mul in (0x2545F4914F6CDD1, 0x369DEA0F31A53F8 | 1):
        h = (h ^ (h >> 29) & 0x7FFFFFFFF) * mul
    k = (h >> 20) & 0xFFFFFF
    if wtype == "f32":
        return (k + 1).to(torch.float32) * (1.0 / (1 << 24))
    return (k * hi >> 24).to(torch.int32) + 1


def _edges(case, gen, dev):
    """(n, u, v): the arcs of the case's graph."""
    f = case["family"]

    def ints(hi, k):
        return torch.randint(0, hi, (k,), generator=gen, device=dev, dtype=torch.int64)

    if f in ("grid", "road"):
        W, H = case["W"], case["H"]
        n = W * H
        ids = torch.arange(n, device=dev, dtype=torch.int64).view(H, W)
        a = torch.cat([ids[:, :-1].reshape(-1), ids[:-1, :].reshape(-1)])
        b = torch.cat([ids[:, 1:].reshape(-1), ids[1:, :].reshape(-1)])
        if f == "road":
            # 5% of the streets missing; highways join 0.5% as many pairs up to 64 blocks apart
            keep = torch.rand(a.numel(), generator=gen, device=dev) >= 0.05
            a, b = a[keep], b[keep]
            k = max(1, a.numel() // 200)
            x, y = ints(W, k), ints(H, k)
            length = ints(63, k) + 2
            dx = torch.minimum(ints(65, k), length)
            sx, sy = ints(2, k) * 2 - 1, ints(2, k) * 2 - 1
            x2 = (x + sx * dx).clamp(0, W - 1)
            y2 = (y + sy * (length - dx)).clamp(0, H - 1)
            a, b = torch.cat([a, y * W + x]), torch.cat([b, y2 * W + x2])
        return n, torch.cat([a, b]), torch.cat([b, a])
    if f == "rmat":
        n, k = 1 << case["scale"], case["ef"] << case["scale"]
        u, v = torch.zeros(k, dtype=torch.int64, device=dev), torch.zeros(k, dtype=torch.int64, device=dev)
        for _ in range(case["scale"]):
            r = torch.rand(k, generator=gen, device=dev)
            u = u * 2 + (r >= 0.76)
            v = v * 2 + ((r >= 0.57) & (r < 0.76) | (r >= 0.95))
        p = torch.randperm(n, generator=gen, device=dev)
        u, v = p[u], p[v]
        return n, torch.cat([u, v]), torch.cat([v, u])
    n, k = case["n"], case["m"]
    u, v = ints(n, k), ints(n, k)
    if f == "er":
        u, v = torch.cat([u, v]), torch.cat([v, u])
    return n, u, v


def _graph(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(seed)
    n, u, v = _edges(case, gen, dev)
    row, col, u = _csr(n, u, v)
    w = _weights(u, col.to(torch.int64), seed + 1, case["hi"], case["wtype"])
    if case["family"] == "road":
        # a highway costs 20 a block, a street 1 to 1000
        W = case["W"]
        c = col.to(torch.int64)
        blocks = (u % W - c % W).abs() + (u // W - c // W).abs()
        w = torch.where(blocks > 1, (20 * blocks).to(torch.int32), w)
    return n, row, col, w, gen


def _sources(row, k, gen):
    """k vertices that have arcs, uniformly."""
    ok = torch.nonzero(row[1:] > row[:-1]).view(-1)
    at = torch.randint(0, ok.numel(), (k,), generator=gen, device=row.device)
    return ok[at].to(torch.int32)


class _Server:
    """The server that a program keeps; it ends before its graph goes."""

    def __init__(self, graph):
        self.graph, self.handle = graph, S.sssp_serve_create()

    def __del__(self):
        S.sssp_serve_destroy(self.handle)


def prepare(case, seed):
    n, row, col, w, gen = _graph(case, seed)
    nq = case.get("nq", 1)
    srcs = _sources(row, nq, gen)
    out = torch.float32 if case["wtype"] == "f32" and case["call"] != "bfs" else torch.int32
    s = {"call": case["call"], "n": n, "src": int(srcs[0]), "srcs": srcs, "sources": srcs.tolist(),
         "dist": torch.empty(nq * n, dtype=out, device="cuda"),
         "pred": torch.empty(nq * n, dtype=torch.int32, device="cuda") if case["pred"] else None}
    if case["call"] == "noalloc":
        s["row"], s["m"] = row, col.numel()
        s["arcs"] = torch.stack([col, w.view(torch.int32)], 1).contiguous()
        s["wtype"] = S.SSSP_W_F32 if case["wtype"] == "f32" else S.SSSP_W_U32
    else:
        s["graph"] = S.Graph(row, col, w, case["wtype"])
    if case["call"] == "serve":
        s["server"] = _Server(s["graph"])
    return s


def run(s):
    d, p, n = s["dist"], s["pred"], s["n"]
    if s["call"] == "solve":
        s["graph"].solve(s["src"], d, p)
    elif s["call"] == "bfs":
        s["graph"].bfs(s["src"], d, p)
    elif s["call"] == "batch":
        s["graph"].solve_batch(s["srcs"], d, p)
    elif s["call"] == "noalloc":
        S.sssp_solve_noalloc(s["row"], s["arcs"], n, s["m"], s["wtype"], s["src"], d, p)
    else:
        h, g = s["server"].handle, s["graph"].handle
        tickets = [S.sssp_serve_submit(h, g, v, d[q * n:(q + 1) * n], None if p is None else p[q * n:(q + 1) * n])
                   for q, v in enumerate(s["sources"])]
        for t in tickets:
            state, code = S.sssp_serve_wait(h, t)
            if state != S.Q_DONE:
                raise S.SsspError(code, "serve")
            S.sssp_serve_release(h, t)
    return {"dist": d} if p is None else {"dist": d, "pred": p}


# ---------------------------------------------------------------- bounds

def _arcs(case):
    """(vertices, arcs) of the case's graph, about."""
    f = case["family"]
    if f in ("grid", "road"):
        return case["W"] * case["H"], 4 * case["W"] * case["H"]
    if f == "rmat":
        return 1 << case["scale"], 2 * case["ef"] << case["scale"]
    return case["n"], case["m"] * (2 if f == "er" else 1)


def work(case):
    """The graph read once (4 B a row, 8 B an arc; a search by hops needs no weights) and the answers
    written once; one addition and one comparison per arc and query."""
    n, m = _arcs(case)
    nq = case.get("nq", 1)
    arc = 4 if case["call"] == "bfs" else 8
    return {"bytes": 4 * n + arc * m + nq * n * (8 if case["pred"] else 4),
            "flops": (1 if case["call"] == "bfs" else 2) * nq * m}


# ---------------------------------------------------------------- the answer in 64 bits

def _relax(row, col, u, w, src, inf):
    """Shortest lengths from src by rounds over the arcs of the vertices that changed."""
    n = row.numel() - 1
    dist = torch.full((n,), inf, dtype=w.dtype, device=w.device)
    dist[src] = 0
    front = torch.tensor([src], device=w.device)
    start, deg = row[:-1].to(torch.int64), (row[1:] - row[:-1]).to(torch.int64)
    while front.numel():
        k = deg[front]
        total = int(k.sum())
        if not total:
            break
        at = torch.repeat_interleave(start[front] - (torch.cumsum(k, 0) - k), k, output_size=total)
        at += torch.arange(total, device=w.device)
        old = dist.clone()
        dist.scatter_reduce_(0, col[at], dist[u[at]] + w[at], "amin")
        front = torch.nonzero(dist < old).view(-1)
    return dist


def exact(case, seed):
    n, row, col, w, gen = _graph(case, seed)
    m, nq = col.numel(), case.get("nq", 1)
    high = case["family"] in ("grid", "road")
    # a few rounds over all arcs for the large graphs, thousands of small ones for the meshes
    if nq * m > (1 << 23 if high else 1 << 29):
        return None
    srcs = _sources(row, nq, gen).tolist()
    col = col.to(torch.int64)
    u = torch.repeat_interleave(torch.arange(n, device=row.device), (row[1:] - row[:-1]).to(torch.int64))
    if case["call"] == "bfs":
        w = torch.ones_like(col)
    real = w.is_floating_point()
    w = w.to(torch.float64 if real else torch.int64)
    inf = math.inf if real else 1 << 40
    dist, pred = [], []
    for s in srcs:
        d = _relax(row, col, u, w, s, inf)
        if case["pred"]:
            # the smallest-numbered tight in-neighbour
            tight = (d[u] + w == d[col]) & (d[u] < inf)
            p = torch.full((n,), n, dtype=torch.int64, device=w.device)
            p.scatter_reduce_(0, col[tight], u[tight], "amin")
            p[p == n] = -1
            p[s] = s
            pred.append(p)
        dist.append(d if real else torch.where(d < inf, d, -1))
    out = {"dist": torch.cat(dist)}
    if case["pred"]:
        out["pred"] = torch.cat(pred)
    return out
