"""The work that users of this library have it do, as cases that can be timed.

Each case is one pass of a program that holds resident graphs and asks for
breadth-first searches through the public entry points (Graph.run,
Graph.run_multiroot, Graph.run_multi, Server).  Graphs are synthetic, of the
families the repository's workloads name (R-MAT with initiator .57/.19/.19/.05
and 16 edges per vertex, Erdos-Renyi, 2D torus, power law), generated on the
GPU from the seed alone.

Levels are a function of the graph and the root.  Parents are one only with
PARENT_MIN_ID: with PARENT_ANY any vertex one level closer may win the claim,
and two passes differ.  So the searches that ask for any parent write both
arrays, as their users have them do, and hand back the levels; those that ask
for the minimum-id parent hand back both.

Fields of a case:
  call     search   one Graph.run per root
           union    one Graph.run_multiroot over a disjoint union, one root per part
           multi    one Graph.run_multi over all roots
           served   a burst of queries to a Server, results in host memory
  graph    rmat | er | torus | powerlaw (`n` vertices: 2^scale for rmat, side^2 for torus)
  n, roots, rows (id | hub: the rows that bottom-up steps scan), layout
  (csr | dcsc), mode (do | td), parents (none | any | min), directed
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1705_04590_gb300 as bfs

DEV = "cuda"
CHUNK = 1 << 26          # edges generated at a time
EDGE_FACTOR = 16         # generated edges per vertex of an R-MAT or power-law graph


def _search(name, graph, n, roots, rows="hub", layout="csr", mode="do", parents="any", directed=False):
    return {"name": name, "call": "search", "graph": graph, "n": n, "roots": roots, "rows": rows, "layout": layout,
            "mode": mode, "parents": parents, "directed": directed}


def listed():
    return [
        # one query on a small graph with the default options: launch and barrier latency
        _search("search_rmat12", "rmat", 1 << 12, 1, rows="id"),
        # reproducible parents (the (select2nd, min) semiring) on a mid-sized graph
        _search("search_rmat20_min_parents", "rmat", 1 << 20, 2, rows="id", parents="min"),
        # the default options at the size the layouts are compared at
        _search("search_rmat24_id_rows", "rmat", 1 << 24, 4, rows="id"),
        # the same family over the hypersparse column-block tiles
        _search("search_rmat22_dcsc", "rmat", 1 << 22, 2, rows="id", layout="dcsc"),
        # a directed graph: top-down over out-rows, bottom-up over the transpose
        _search("search_rmat24_directed", "rmat", 1 << 24, 2, rows="id", directed=True),
        # the headline: the largest graph, hub-first rows, both outputs
        _search("search_rmat26_hub", "rmat", 1 << 26, 4),
        # no hubs and a vertex count that is a multiple of nothing
        _search("search_er_40m", "er", 40_000_003, 2),
        # thousands of small levels
        _search("search_torus4096", "torus", 4096 * 4096, 1),
        # batched: 64 searches as lane masks in one launch
        {"name": "multi_rmat22", "call": "multi", "graph": "rmat", "n": 1 << 22, "roots": 64, "rows": "hub",
         "parents": "none"},
        # a batch that does not fill its lanes, with minimum-id parents
        {"name": "multi_rmat18_parents", "call": "multi", "graph": "rmat", "n": 1 << 18, "roots": 40, "rows": "id",
         "parents": "min"},
        # an uneven batch of many graphs in one launch
        {"name": "union_256_rmat", "call": "union", "graph": "rmat", "parts": 256, "scale_lo": 10, "scale_hi": 20},
        # a burst of queries to resident graphs of uneven size, a large-diameter one among them
        {"name": "served_burst", "call": "served", "graphs": "rmat:65536,rmat:262144,rmat:1048576,rmat:4194304,"
         "torus:262144", "queries": 40},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["small", "rmat", "min", "td", "dcsc", "directed", "er", "powerlaw", "torus", "multi", "union",
                       "served"])
    if kind == "small":
        return {k: v for k, v in _search("", rng.choice(["er", "powerlaw"]), _log_uniform(rng, 500, 60_000),
                                         1, rows=rng.choice(["id", "hub"])).items() if k != "name"}
    if kind == "multi":
        g = rng.choice(["rmat", "er", "powerlaw"])
        par = rng.choice(["none", "none", "min"])
        most = 18 if par == "min" else 20
        n = 1 << rng.randint(12, most) if g == "rmat" else _log_uniform(rng, 4000, 1 << (most - 1))
        return {"call": "multi", "graph": g, "n": n, "roots": rng.randint(2, 100 if par == "none" else 40), "rows": rng.choice(["id", "hub"]),
                "parents": par}
    if kind == "union":
        lo = rng.randint(8, 12)
        return {"call": "union", "graph": "rmat", "parts": _log_uniform(rng, 16, 160), "scale_lo": lo,
                "scale_hi": rng.randint(lo + 2, 18)}
    if kind == "served":
        gs = [f"rmat:{1 << rng.randint(12, 21)}" for _ in range(rng.randint(1, 3))]
        gs.append(f"er:{_log_uniform(rng, 10_000, 2_000_000)}")
        return {"call": "served", "graphs": ",".join(gs), "queries": rng.randint(4, 60)}
    if kind == "torus":
        side = _log_uniform(rng, 60, 2000)
        c = _search("", "torus", side * side, 1, rows=rng.choice(["id", "hub"]), parents=rng.choice(["any", "min"]))
        if c["parents"] == "min":
            c["rows"] = "id"
    elif kind == "rmat":
        c = _search("", "rmat", 1 << rng.randint(14, 25), rng.randint(1, 4))
    elif kind == "min":
        c = _search("", rng.choice(["rmat", "er", "powerlaw"]), _log_uniform(rng, 20_000, 1_000_000), 1, rows="id",
                    parents="min")
    elif kind == "td":
        c = _search("", rng.choice(["rmat", "er"]), _log_uniform(rng, 100_000, 8_000_000), 1, rows="id", mode="td")
    elif kind == "dcsc":
        c = _search("", rng.choice(["rmat", "er"]), _log_uniform(rng, 30_000, 4_000_000), 1, rows="id", layout="dcsc",
                    mode=rng.choice(["do", "do", "td"]), parents=rng.choice(["any", "min"]))
    elif kind == "directed":
        c = _search("", rng.choice(["rmat", "er"]), _log_uniform(rng, 30_000, 8_000_000), 2, rows="id", directed=True)
    else:
        c = _search("", kind, _log_uniform(rng, 100_000, 20_000_000), 2, rows=rng.choice(["id", "hub"]))
    if c["graph"] == "rmat":
        c["n"] = 1 << int(round(math.log2(c["n"])))
    return {k: v for k, v in c.items() if k != "name"}


# ------------------------------------------------------------------ inputs

def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(0x5EED + 7919 * int(seed))
    return g


def _relabel(gen, n, ids):
    """The vertex ids through one random bijection of [0, n)."""
    label = torch.randperm(n, generator=gen, device=DEV).to(torch.int32)
    return [torch.index_select(label, 0, x) for x in ids]


def _rmat_edges(gen, scale):
    a, b, c = 0.57, 0.19, 0.19
    m = EDGE_FACTOR << scale
    src = torch.empty(m, dtype=torch.int32, device=DEV)
    dst = torch.empty(m, dtype=torch.int32, device=DEV)
    for lo in range(0, m, CHUNK):
        s, d = src[lo:lo + CHUNK], dst[lo:lo + CHUNK]
        s.zero_()
        d.zero_()
        for _ in range(scale):
            r = torch.rand(s.numel(), generator=gen, device=DEV)
            s.mul_(2).add_(r >= a + b)
            d.mul_(2).add_(((r >= a) & (r < a + b)) | (r >= a + b + c))
    return src, dst


def _powerlaw_ends(gen, n, m, gamma=2.1, i0=50.0):
    """Vertex ranks drawn with density proportional to (x + i0)^(-1/(gamma-1)) over [0, n)."""
    e = 1.0 - 1.0 / (gamma - 1.0)
    u = torch.rand(m, generator=gen, device=DEV, dtype=torch.float64)
    x = (u * ((n + i0) ** e - i0 ** e) + i0 ** e) ** (1.0 / e) - i0
    return x.clamp_(0, n - 1).to(torch.int32)


def _edges(gen, graph, n):
    """(src, dst) int32 device arrays: an undirected graph's edges, each once (or a directed one's)."""
    if graph == "rmat":
        src, dst = _rmat_edges(gen, n.bit_length() - 1)
    elif graph == "er":
        # expected degree 16
        return (torch.randint(0, n, (8 * n,), generator=gen, device=DEV, dtype=torch.int32),
                torch.randint(0, n, (8 * n,), generator=gen, device=DEV, dtype=torch.int32))
    elif graph == "powerlaw":
        src, dst = _powerlaw_ends(gen, n, EDGE_FACTOR * n), _powerlaw_ends(gen, n, EDGE_FACTOR * n)
    else:
        side = math.isqrt(n)
        v = torch.arange(n, device=DEV, dtype=torch.int32)
        x, y = v % side, v // side
        src = torch.cat([v, v])
        dst = torch.cat([y * side + (x + 1) % side, ((y + 1) % side) * side + x])
    return _relabel(gen, n, (src, dst))


def _union_scales(case):
    """The parts' scales: the mix of sizes belongs to the case, the graphs to the seed."""
    sizes = random.Random(4242)
    return [sizes.randint(case["scale_lo"], case["scale_hi"]) for _ in range(case["parts"])]


def _union_edges(gen, case):
    """The parts' edges with their ids offset, the parts' first ids, and the vertex count."""
    src, dst, first, n = [], [], [], 0
    for sc in _union_scales(case):
        s, d = _relabel(gen, 1 << sc, _rmat_edges(gen, sc))
        src.append(s + n)
        dst.append(d + n)
        first.append(n)
        n += 1 << sc
    return torch.cat(src), torch.cat(dst), first, n


def _with_edges(src, dst, n, directed=False):
    """Which vertices have an edge (an outgoing one when directed) to another vertex."""
    has = torch.zeros(n, dtype=torch.bool, device=DEV)
    for lo in range(0, src.numel(), CHUNK):
        s, d = src[lo:lo + CHUNK], dst[lo:lo + CHUNK]
        keep = s != d
        has[s[keep].long()] = True
        if not directed:
            has[d[keep].long()] = True
    return has


def _roots(gen, src, dst, n, k, directed=False):
    """k roots, uniform over the vertices with an edge."""
    ids = _with_edges(src, dst, n, directed).nonzero().flatten()
    return ids[torch.randint(0, ids.numel(), (k,), generator=gen, device=DEV)].tolist()


def _inputs(case, seed):
    """What the searches run on: a list of (src, dst, n, roots), one per graph."""
    gen = _generator(seed)
    if case["call"] == "served":
        out = []
        for i, spec in enumerate(case["graphs"].split(",")):
            kind, n = spec.split(":")
            src, dst = _edges(gen, kind, int(n))
            k = len(range(i, case["queries"], len(case["graphs"].split(","))))
            out.append((src, dst, int(n), _roots(gen, src, dst, int(n), k)))
        return out
    if case["call"] == "union":
        src, dst, first, n = _union_edges(gen, case)
        has = _with_edges(src, dst, n)
        roots = []
        for i, lo in enumerate(first):
            hi = first[i + 1] if i + 1 < len(first) else n
            ids = has[lo:hi].nonzero().flatten()
            roots.append(lo + int(ids[torch.randint(0, ids.numel(), (1,), generator=gen, device=DEV)]))
        return [(src, dst, n, roots)]
    src, dst = _edges(gen, case["graph"], case["n"])
    return [(src, dst, case["n"], _roots(gen, src, dst, case["n"], case["roots"], case.get("directed", False)))]


def _options(case):
    return bfs.options(mode=bfs.MODE_TD_ONLY if case.get("mode") == "td" else bfs.MODE_DO,
                       layout=bfs.LAYOUT_DCSC_TILED if case.get("layout") == "dcsc" else bfs.LAYOUT_CSR,
                       parent_mode=bfs.PARENT_MIN_ID if case["call"] == "search" and case["parents"] == "min"
                       else bfs.PARENT_ANY,
                       bu_rows=bfs.BU_ROWS_HUB_FIRST if case.get("rows") == "hub" else bfs.BU_ROWS_BY_ID)


def prepare(case, seed):
    """Resident graphs, the roots to search from and the output arrays."""
    parts = _inputs(case, seed)
    if case["call"] == "served":
        graphs = [bfs.Graph.from_edges(s, d, n) for s, d, n, _ in parts]
        server = bfs.Server(hbm_budget_bytes=24 << 30, max_lanes=64)
        queries = []
        for g, (_, _, n, roots) in zip(graphs, parts):
            slot = server.add_graph(g)
            queries += [(i, slot, r, torch.empty(n, dtype=torch.int32, pin_memory=True).numpy())
                        for i, r in enumerate(roots)]
        queries.sort(key=lambda q: q[:2])      # the graphs in turn
        return {"call": "served", "server": server, "graphs": graphs, "queries": [q[1:] for q in queries]}
    (src, dst, n, roots), = parts
    graph = bfs.Graph.from_edges(src, dst, n, dcsc=case.get("layout") == "dcsc", hub_first=case.get("rows") == "hub",
                                 directed=case.get("directed", False))
    state = {"call": case["call"], "graph": graph, "opts": _options(case) if case["call"] != "union" else None,
             "min": case.get("parents") == "min"}
    new = lambda k: torch.empty(k, dtype=torch.int32, device=DEV)  # noqa: E731
    if case["call"] == "search":
        state |= {"roots": roots, "level": [new(n) for _ in roots],
                  "parent": [new(n) if case["parents"] != "none" else None for _ in roots]}
    else:
        k = len(roots) if case["call"] == "multi" else 1
        state |= {"roots": np.array(roots, np.int32), "level": new(k * n),
                  "parent": new(k * n) if state["min"] else None}
    return state


def run(state):
    if state["call"] == "served":
        server = state["server"]
        tickets = [server.submit(slot, root, out) for slot, root, out in state["queries"]]
        for t in tickets:
            if not server.wait(t, 60_000):
                raise RuntimeError("a query did not complete within a minute")
        return [out for _, _, out in state["queries"]]
    g = state["graph"]
    if state["call"] == "search":
        for root, level, parent in zip(state["roots"], state["level"], state["parent"]):
            g.run(root, parent=parent, level=level, opts=state["opts"])
    elif state["call"] == "union":
        g.run_multiroot(state["roots"], level=state["level"])
    else:
        g.run_multi(state["roots"], state["level"], parent=state["parent"], opts=state["opts"])
    return {"level": state["level"], "parent": state["parent"]} if state["min"] else {"level": state["level"]}


# ------------------------------------------------------------------ what a pass needs

def _sizes(case):
    """(vertices, stored column ids, searches) of each graph, from the case alone."""
    def ids(graph, n):
        return {"rmat": 2 * EDGE_FACTOR, "er": 16, "torus": 4, "powerlaw": 2 * EDGE_FACTOR}[graph] * n
    if case["call"] == "served":
        specs = [s.split(":") for s in case["graphs"].split(",")]
        return [(int(n), ids(k, int(n)), len(range(i, case["queries"], len(specs))))
                for i, (k, n) in enumerate(specs)]
    if case["call"] == "union":
        n = sum(1 << sc for sc in _union_scales(case))
        return [(n, ids("rmat", n), 1)]
    return [(case["n"], ids(case["graph"], case["n"]), case["roots"])]


def work(case):
    """Per search: each output written once and one neighbour id per vertex read (what a
    bottom-up step that always hits at once would read); a top-down-only search reads every
    row, and so does a batch (once for all its searches)."""
    total = 0
    for n, nnz, k in _sizes(case):
        outs = 2 if case.get("parents", "none") != "none" else 1
        rows = 4 * nnz + 8 * n
        if case["call"] == "multi":
            total += 4 * n * outs * k + rows
        else:
            total += k * (4 * n * outs + (rows if case.get("mode") == "td" else 4 * n))
    return {"bytes": total, "flops": 0}


# ------------------------------------------------------------------ the same answers in plain torch

def _levels(src, dst, n, roots):
    """Hop distance to the nearest root along src -> dst, -1 if there is no path."""
    level = torch.full((n,), -1, dtype=torch.int32, device=DEV)
    level[torch.tensor(roots, device=DEV)] = 0
    d = 0
    while True:
        found = False
        for lo in range(0, src.numel(), 1 << 28):
            s, t = src[lo:lo + (1 << 28)], dst[lo:lo + (1 << 28)]
            hit = t[(torch.index_select(level, 0, s) == d) & (torch.index_select(level, 0, t) == -1)]
            if hit.numel():
                level[hit.long()] = d + 1
                found = True
        if not found:
            return level
        d += 1


def _min_parents(src, dst, n, level, root):
    """The smallest u one level closer with an edge u -> v; the root its own; -1 where not reached."""
    up = (torch.index_select(level, 0, src) == torch.index_select(level, 0, dst) - 1) & \
        (torch.index_select(level, 0, src) >= 0)
    big = torch.full((n,), 2 ** 31 - 1, dtype=torch.int32, device=DEV)
    big.scatter_reduce_(0, dst[up].long(), src[up], "amin")
    big[big == 2 ** 31 - 1] = -1
    big[root] = root
    return big


def exact(case, seed):
    if case.get("graph") == "torus" and case["n"] > 1 << 20:
        return None      # thousands of passes over all edges
    parts = []
    for src, dst, n, roots in _inputs(case, seed):
        if not case.get("directed"):
            src, dst = torch.cat([src, dst]), torch.cat([dst, src])
        parts.append((src, dst, n, roots))
    if case["call"] == "served":
        out = []
        for slot, (src, dst, n, roots) in enumerate(parts):
            out += [(i, slot, _levels(src, dst, n, [r])) for i, r in enumerate(roots)]
        out.sort(key=lambda q: q[:2])
        return [lv.cpu().numpy() for _, _, lv in out]
    (src, dst, n, roots), = parts
    if case["call"] == "union":
        return {"level": _levels(src, dst, n, roots)}
    level = [_levels(src, dst, n, [r]) for r in roots]
    parent = [_min_parents(src, dst, n, lv, r) for lv, r in zip(level, roots)] if case["parents"] == "min" else None
    if case["call"] == "multi":
        level = torch.cat(level)
        parent = torch.cat(parent) if parent else None
    return {"level": level, "parent": parent} if parent is not None else {"level": level}
