"""Timed cases of the mapping library: what its users call, over the sizes they call it with.

A case is one call sequence of ``paper_2510_12196_gb300.gpumap``.  ``call`` says which:

- ``map``:       the mapping of a new graph, from its CSR to the PE of every vertex: ``map_create``
                 (which copies and validates the CSR), ``map_run`` or ``map_run_hm``, ``map_destroy``.
                 ``inputs``: ``device`` (CSR tensors on the GPU) or ``host`` (numpy arrays).
- ``remap``:     ``map_run`` on a context that the program keeps.
- ``refine``:    a mapping that the program has is set, refined by a fixed number of Alg. 6 rounds and
                 read back, on a context that it keeps.
- ``batch``:     the same for many graphs in one ``map_batch``.
- ``serve``:     a burst of mapping requests through a ``MapServer`` that the program keeps.
- ``objective``: ``map_objective_noalloc``, the cost of a mapping that lies in device memory.

Graphs are the library's workload families, drawn on the GPU: 2D / 3D grids, random geometric graphs
(ids in cell order, edge weights 1..wmax), R-MAT graphs ((.57, .19, .19, .05), duplicates and
self-loops dropped, relabelled).  All outputs are whole numbers: the PE of each vertex and J.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2510_12196_gb300 import gpumap as G
from paper_2510_12196_gb300 import inputs as I

_DIST = (1, 10, 100, 1000)


def listed():
    return [
        # the smallest call: ten rounds on a small grid; launches and round trips are all it costs
        dict(name="refine_grid64", call="refine", graph="grid", nx=64, ny=64, nz=1, hier="4:8", rounds=10),
        # small mapping requests from host arrays: a 3D stencil, and an odd size with vertex weights on a
        # machine whose counts are no powers of two
        dict(name="map_grid16", call="map", graph="grid", nx=16, ny=16, nz=16, hier="4:8", inputs="host"),
        dict(name="map_rgg_50021", call="map", graph="rgg", n=50021, degree=12, wmax=10, vwmax=4, hier="4:8:6",
             inputs="host"),
        # ordinary meshes: a random geometric graph of 2^20 vertices, the largest 3D stencil of the serving mix
        dict(name="map_rgg_2e20", call="map", graph="rgg", n=1 << 20, degree=12, wmax=10, vwmax=1, hier="4:8:8",
             inputs="device"),
        dict(name="map_grid128", call="map", graph="grid", nx=128, ny=128, nz=128, hier="4:16:16", inputs="device"),
        # power-law graphs: an odd ordinary size, and the largest, re-mapped on a kept context
        dict(name="map_rmat_200003", call="map", graph="rmat", n=200003, factor=16, hier="4:16", inputs="device"),
        dict(name="remap_rmat_2e22", call="remap", graph="rmat", n=1 << 22, factor=16, hier="4:16:8"),
        # the variants: matching coarsener with J-gain rebalancing, and hierarchical multisection
        dict(name="map_rgg_2e18_match", call="map", graph="rgg", n=1 << 18, degree=12, wmax=10, vwmax=1,
             hier="4:8:8", inputs="device", coarsener=1, reb_objective=1),
        dict(name="hm_rgg_2e17", call="map", graph="rgg", n=1 << 17, degree=12, wmax=10, vwmax=1, hier="4:8:4",
             inputs="device", hm=True),
        # many graphs of uneven size at once: ten rounds each in one batch, and a burst of requests
        dict(name="batch_24", call="batch", count=24, lo=1 << 12, hi=1 << 18, rounds=10),
        dict(name="serve_16", call="serve", count=16, lo=1 << 10, hi=1 << 17),
        # the cost of a given mapping
        dict(name="objective_rmat_2e20", call="objective", graph="rmat", n=1 << 20, factor=16, hier="4:16:8"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_graph(rng, lo, hi):
    n = _log_uniform(rng, lo, hi)
    family = rng.choice(("rgg", "grid", "rmat"))
    if family == "rgg":
        return dict(graph="rgg", n=n, degree=rng.choice((10, 12)), wmax=rng.choice((1, 10)), vwmax=rng.choice((1, 4)))
    if family == "grid":
        nx = max(2, int(round(n ** (1 / 3) * rng.uniform(0.6, 1.6))))
        ny = max(2, int(round(math.sqrt(n / nx))))
        return dict(graph="grid", nx=nx, ny=ny, nz=max(1, n // (nx * ny)))
    return dict(graph="rmat", n=n, factor=rng.choice((8, 16)))


def draw(rng):
    call = rng.choice(("map", "map", "map", "remap", "refine", "batch", "serve", "objective"))
    if call == "batch":
        return dict(call=call, count=rng.randint(8, 32), lo=1 << 12, hi=_log_uniform(rng, 1 << 14, 1 << 18), rounds=10)
    if call == "serve":
        return dict(call=call, count=rng.randint(8, 24), lo=1 << 10, hi=_log_uniform(rng, 1 << 13, 1 << 18))
    hier = rng.choice(("4:8", "4:8:6", "4:8:8", "4:16:8", "4:16:16", "2:4:16:8"))
    if call == "refine":
        return dict(call=call, hier=hier, rounds=10, **_draw_graph(rng, 1 << 12, 1 << 18))
    if call == "objective":
        return dict(call=call, hier=hier, **_draw_graph(rng, 1 << 14, 1 << 21))
    if call == "remap":
        return dict(call=call, hier=hier, **_draw_graph(rng, 1 << 15, 1 << 21))
    case = dict(call=call, hier=hier, inputs=rng.choice(("host", "device")), **_draw_graph(rng, 1 << 11, 1 << 20))
    if rng.random() < 0.2:
        case.update(coarsener=1, reb_objective=1)
    return case


# ---------------------------------------------------------------------------
# graphs, drawn on the GPU: (n, xadj int64, adj int32, weights int32, vertex weights int32)
# ---------------------------------------------------------------------------

def _mix(z):
    """SplitMix64's output function on int64 tensors (logical shifts)."""
    z = z - 0x61C8864680B583EB
    z = (z ^ ((z >> 30) & ((1 << 34) - 1))) * -0x40A7B892E31B1A47
    z = (z ^ ((z >> 27) & ((1 << 37) - 1))) * -0x6B2FB644ECCEEE15
    return (z ^ ((z >> 31) & ((1 << 33) - 1))) & ((1 << 63) - 1)


def _csr(n, u, v, seed, wmax=1, vwmax=1):
    key = torch.sort(torch.cat([u * n + v, v * n + u])).values
    src = key // n
    adj = key - src * n
    xadj = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    xadj[1:] = torch.cumsum(torch.bincount(src, minlength=n), 0)
    if wmax > 1:
        w = (_mix((torch.minimum(src, adj) * n + torch.maximum(src, adj)) ^ seed) % wmax + 1).to(torch.int32)
    else:
        w = torch.ones(key.numel(), dtype=torch.int32, device="cuda")
    ids = torch.arange(n, dtype=torch.int64, device="cuda")
    vw = (_mix(ids ^ (seed + 77)) % vwmax + 1).to(torch.int32)
    return n, xadj, adj.to(torch.int32), w, vw


def _grid(nx, ny, nz, seed):
    ids = torch.arange(nx * ny * nz, dtype=torch.int64, device="cuda").reshape(nz, ny, nx)
    ends = [(ids[:, :, :-1], ids[:, :, 1:]), (ids[:, :-1], ids[:, 1:]), (ids[:-1], ids[1:])]
    return _csr(nx * ny * nz, torch.cat([a.reshape(-1) for a, _ in ends]), torch.cat([b.reshape(-1) for _, b in ends]),
                seed)


def _rgg(n, degree, wmax, vwmax, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    r = math.sqrt(degree / (math.pi * n))
    side = max(1, int(1.0 / r))
    p = torch.rand(n, 2, generator=gen, device="cuda", dtype=torch.float64)
    c = torch.clamp((p * side).to(torch.int64), max=side - 1)
    order = torch.argsort(c[:, 1] * side + c[:, 0], stable=True)
    p, c = p[order], c[order]
    count = torch.bincount(c[:, 1] * side + c[:, 0], minlength=side * side)
    start = torch.cumsum(count, 0) - count
    us, vs = [], []
    for dx, dy in ((0, 0), (1, 0), (-1, 1), (0, 1), (1, 1)):
        cx, cy = c[:, 0] + dx, c[:, 1] + dy
        src = torch.nonzero((cx >= 0) & (cx < side) & (cy < side)).reshape(-1)
        cell = (cy * side + cx)[src]
        k = count[cell]
        u = torch.repeat_interleave(src, k)
        v = torch.repeat_interleave(start[cell] - (torch.cumsum(k, 0) - k), k) + torch.arange(u.numel(), device="cuda")
        near = ((p[u] - p[v]) ** 2).sum(1) < r * r
        if dx == 0 and dy == 0:
            near &= u < v
        us.append(u[near])
        vs.append(v[near])
    return _csr(n, torch.cat(us), torch.cat(vs), seed, wmax, vwmax)


def _rmat(n, factor, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    bits, keys, left = max(1, (n - 1).bit_length()), [], factor * n
    while left:
        s = min(left, 1 << 24)
        u = torch.zeros(s, dtype=torch.int64, device="cuda")
        v = torch.zeros(s, dtype=torch.int64, device="cuda")
        for _ in range(bits):
            x = torch.rand(s, generator=gen, device="cuda")
            u = 2 * u + (x >= 0.76)
            v = 2 * v + (((x >= 0.57) & (x < 0.76)) | (x >= 0.95))
        keep = (u != v) & (u < n) & (v < n)
        u, v = u[keep], v[keep]
        keys.append(torch.minimum(u, v) * n + torch.maximum(u, v))
        left -= s
    key = torch.sort(torch.cat(keys)).values
    key = key[torch.cat([torch.ones(1, dtype=torch.bool, device="cuda"), key[1:] != key[:-1]])]
    perm = torch.randperm(n, generator=gen, device="cuda")
    return _csr(n, perm[key // n], perm[key % n], seed)


def _graph(case, seed):
    if case["graph"] == "grid":
        return _grid(case["nx"], case["ny"], case["nz"], seed)
    if case["graph"] == "rgg":
        return _rgg(case["n"], case["degree"], case["wmax"], case["vwmax"], seed)
    return _rmat(case["n"], case["factor"], seed)


def _host(g):
    n, xadj, adj, w, vw = g
    return I.Graph(n, *(a.cpu().numpy() for a in (xadj, adj, w, vw)))


def _mapping(n, k, seed):
    return (_mix(torch.arange(n, dtype=torch.int64, device="cuda") ^ (seed + 5)) % k).to(torch.int32)


def _machine(hier):
    h = tuple(int(a) for a in hier.split(":"))
    return h, _DIST[:len(h)]


def _items(case, seed):
    """The graphs of a batch or a burst: sizes and machines spread alike for every seed."""
    for i in range(case["count"]):
        u = (i * 0.6180339887498949) % 1.0
        n = int(round(case["lo"] * (case["hi"] / case["lo"]) ** u))
        if case["call"] == "batch":
            yield dict(graph="rgg", n=n, degree=10, wmax=10, vwmax=1), ("4:8", "4:8:8", "2:4:16:8")[i % 3], seed + i
        elif i % 2:
            nx = max(2, round(n ** (1 / 3)))
            yield dict(graph="grid", nx=nx, ny=nx, nz=max(1, n // (nx * nx))), ("4:8", "4:8:8")[i // 2 % 2], seed + i
        else:
            yield dict(graph="rgg", n=n, degree=12, wmax=10, vwmax=1), ("4:8", "4:16:8", "4:16:16")[i // 2 % 3], seed + i


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------

class _Batch:
    """A batch and its contexts, given back in order."""

    def __init__(self, mappers, rounds):
        self.mappers = mappers
        self.handle = G.map_batch_create([m.ctx for m in mappers], G.map_batch_opts_default(rounds=rounds))

    def __del__(self):
        G.map_batch_destroy(self.handle)
        for m in self.mappers:
            m.close()


class _Server(G.MapServer):
    def __del__(self):
        self.close()


def _config(case, seed):
    cfg = G.map_config_default(seed)
    cfg.coarsener = case.get("coarsener", 0)
    cfg.reb_objective = case.get("reb_objective", 0)
    return cfg


def prepare(case, seed):
    call = case["call"]
    if call == "batch":
        mappers, pis = [], []
        for c, hier, s in _items(case, seed):
            g = _graph(c, s)
            h, d = _machine(hier)
            mappers.append(G.Mapper(I.Graph(g[0], *g[1:]), h, d, cfg=_config(case, s), device_inputs=g[1:]))
            pis.append(_mapping(g[0], math.prod(h), s).cpu().numpy())
        return dict(call=call, batch=_Batch(mappers, case["rounds"]), pis=pis)
    if call == "serve":
        jobs = []
        for c, hier, s in _items(case, seed):
            g = _host(_graph(c, s))
            jobs.append((g, *_machine(hier), _config(case, s), np.zeros(g.n, np.int32)))
        return dict(call=call, server=_Server(), jobs=jobs)
    g = _graph(case, seed)
    h, d = _machine(case["hier"])
    state = dict(call=call, hier=h, dist=d, n=g[0])
    if call == "objective":
        return dict(state, csr=g[1:], pi=_mapping(g[0], math.prod(h), seed),
                    out=torch.zeros(2, dtype=torch.int64, device="cuda"))
    state["pi"] = np.zeros(g[0], np.int32)
    if call == "map":
        graph, csr = (_host(g), None) if case["inputs"] == "host" else (I.Graph(g[0], *g[1:]), g[1:])
        return dict(state, graph=graph, csr=csr, cfg=_config(case, seed), hm=case.get("hm", False))
    state["mapper"] = G.Mapper(I.Graph(g[0], *g[1:]), h, d, cfg=_config(case, seed), device_inputs=g[1:])
    if call == "refine":
        state.update(pi=_mapping(g[0], math.prod(h), seed).cpu().numpy(), rounds=case["rounds"])
    return state


def run(state):
    call = state["call"]
    if call == "map":
        with G.Mapper(state["graph"], state["hier"], state["dist"], cfg=state["cfg"],
                      device_inputs=state["csr"]) as m:
            J = (G.map_run_hm if state["hm"] else G.map_run)(m.ctx, state["pi"])
        return {"pi": state["pi"], "J": J}
    if call == "remap":
        return {"J": G.map_run(state["mapper"].ctx, state["pi"]), "pi": state["pi"]}
    if call == "refine":
        ctx = state["mapper"].ctx
        G.map_set_mapping(ctx, 0, state["pi"])
        J, weight, rounds = G.map_refine(ctx, 0, state["rounds"])
        return {"J": J, "weight": weight, "rounds": rounds, "pi": G.map_get_mapping(ctx, 0)}
    if call == "batch":
        b = state["batch"]
        for m, pi in zip(b.mappers, state["pis"]):
            G.map_set_mapping(m.ctx, 0, pi)
        G.map_batch_launch(b.handle)
        J, weight, rounds = G.map_batch_results(b.handle, len(b.mappers))
        return {"J": J, "weight": weight, "rounds": rounds, "pi": [G.map_get_mapping(m.ctx, 0) for m in b.mappers]}
    if call == "serve":
        server = state["server"]
        tickets = [server.submit(g, h, d, cfg=cfg, out_pi=pi) for g, h, d, cfg, pi in state["jobs"]]
        done = [server.wait(t) for t in tickets]
        return {"status": [r.status for r, _ in done], "J": np.array([r.J for r, _ in done]), "pi": [p for _, p in done]}
    G.map_objective_noalloc(*state["csr"], state["n"], state["pi"], state["hier"], state["dist"], state["out"])
    return state["out"]


def _size(c):
    """Vertices and CSR entries (grids exactly, the random families as expected)."""
    if c["graph"] == "grid":
        x, y, z = c["nx"], c["ny"], c["nz"]
        return x * y * z, 2 * ((x - 1) * y * z + x * (y - 1) * z + x * y * (z - 1))
    return c["n"], c["n"] * (c["degree"] if c["graph"] == "rgg" else int(1.8 * c["factor"]))


def work(case):
    """The CSR and the vertex weights read once, the mapping written once (read, too, where it is given)."""
    graphs = [c for c, _, _ in _items(case, 0)] if "graph" not in case else [case]
    moved = 0
    for c in graphs:
        n, m = _size(c)
        moved += 8 * (n + 1) + 8 * m + 8 * n + (4 * n if case["call"] in ("refine", "batch") else 0)
    return {"bytes": moved, "flops": 0}


def exact(case, seed):
    """J and the largest block weight of a given mapping; a map itself has no such value."""
    if case["call"] != "objective":
        return None
    n, xadj, adj, w, vw = _graph(case, seed)
    h, d = _machine(case["hier"])
    pi = _mapping(n, math.prod(h), seed).to(torch.int64)
    p, q = torch.repeat_interleave(pi, xadj[1:] - xadj[:-1]), pi[adj.to(torch.int64)]
    dist, below = torch.zeros_like(p), 1
    for a, di in zip(h, d):  # the smallest level whose group holds both
        dist = torch.where(p // below != q // below, di, dist)
        below *= a
    block = torch.zeros(math.prod(h), dtype=torch.int64, device="cuda").index_add_(0, pi, vw.to(torch.int64))
    return torch.stack([(dist * w).sum(), block.max()])
