"""Calls that stand for this library's use, each through its public binding, with their inputs.

A case is a dict of plain values.  `algo` names the call, `graph` the family (`rmat`: power-law, `grid`: road-like
lattice, both by the recipes of the workloads in bench.py, drawn here on the GPU from the seed), `n` or `w` x `h` the
size (an RMAT graph of any n: 16 n samples of the next power of two, folded onto n ids), `k` the sources of a batch,
`source` where a single query starts.  Queries run on a graph that is already loaded, except `new_graph`.
"""
import math

import numpy as np
import torch

from paper_2012_07990_gb300 import g2

EDGE_FACTOR = 16
DAMPING, ROUNDS = 0.85, 20
RMAT_WMAX, GRID_WMAX = 255, 1000   # weight ranges of the batched RMAT and the road workloads


def listed():
    return [
        # the smallest query: one BFS on a small power-law graph, where launches and latency count
        dict(name="bfs_rmat14", algo="bfs", graph="rmat", n=1 << 14, source="hub", parent=True),
        # social-network-sized single queries, as the benchmark's step runs them
        dict(name="bfs_rmat22", algo="bfs", graph="rmat", n=1 << 22, source="hub", parent=True),
        dict(name="cc_rmat22", algo="cc", graph="rmat", n=1 << 22),
        dict(name="pagerank_rmat22", algo="pagerank", graph="rmat", n=1 << 22),
        # a graph seen for the first time: upload from pinned host memory, PageRank's layouts, 20 rounds, release
        dict(name="new_graph_n700001", algo="new_graph", graph="rmat", n=700001),
        # a route query's breadth-first search on a city-sized road network (hundreds of small levels)
        dict(name="bfs_grid1024", algo="bfs", graph="grid", w=1024, h=1024, source="corner", parent=True),
        # shortest paths over a continent-sized road network
        dict(name="sssp_grid4096", algo="sssp", graph="grid", w=4096, h=4096, source="corner", delta=16384),
        # a served shortest-path query on a power-law graph of a ragged size
        dict(name="sssp_rmat_n1300003", algo="sssp", graph="rmat", n=1300003, source="random", delta=64),
        # queries batched on one graph, as the server issues them at load
        dict(name="bfs_batch64_rmat21", algo="bfs_batch", graph="rmat", n=1 << 21, k=64),
        dict(name="sssp_batch32_rmat21", algo="sssp_batch", graph="rmat", n=1 << 21, k=32, delta=64),
        # centrality from a sample of sources
        dict(name="bc16_rmat21", algo="bc", graph="rmat", n=1 << 21, k=16),
        # a caller's own loop: one operator over a frontier of a twentieth of the vertices, ETWC as the paper has it
        dict(name="apply_relax_rmat20", algo="apply", graph="rmat", n=1 << 20, lb="ETWC", share=0.05),
    ]


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    algo = rng.choice(["bfs", "bfs", "cc", "pagerank", "new_graph", "sssp", "sssp", "bfs_batch", "sssp_batch", "bc",
                       "apply"])
    batch = algo in ("bfs_batch", "sssp_batch", "bc")
    grid = algo not in ("new_graph", "apply") and rng.random() < 0.35
    case = dict(algo=algo, graph="grid" if grid else "rmat")
    if grid:
        top = 400 if batch else 2000
        case.update(w=spread(40, top), h=spread(40, top))
    else:
        case.update(n=spread(1 << 10, 1 << (20 if batch else 21 if algo == "sssp" else 22)))
    if algo == "bfs":
        case.update(source=rng.choice(["corner", "random"] if grid else ["hub", "random"]), parent=rng.random() < 0.7)
    if algo == "sssp":
        case.update(source="random")
    if algo in ("sssp", "sssp_batch"):
        case.update(delta=spread(1024, 16384) if grid else spread(16, 512))
    if batch:
        case.update(k=rng.randint(2, {"bfs_batch": 64, "sssp_batch": 32, "bc": 16}[algo]))
    if algo == "apply":
        case.update(lb=rng.choice(["VERTEX_BASED", "CM", "WM", "STRICT", "ETWC", "TWC"]),
                    share=round(math.exp(rng.uniform(math.log(0.002), math.log(0.5))), 4))
        if case["lb"] == "VERTEX_BASED":
            case["n"] = min(case["n"], 1 << 17)   # a thread walks a hub's whole list: only small graphs use it
    return case


# ------------------------------------------------------------------------------------------------ inputs
def _csr(n, u, v):
    """Symmetric CSR (int32, lists ascending, no loops, no duplicates) of the pairs (u, v)."""
    keep = u != v
    u, v = u[keep], v[keep]
    key = torch.unique(torch.cat([u * n + v, v * n + u]))
    src = torch.div(key, n, rounding_mode="floor")
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=key.device)
    rowptr[1:] = torch.cumsum(torch.bincount(src, minlength=n), 0)
    return rowptr.to(torch.int32), (key - src * n).to(torch.int32)


def _rmat(n, gen):
    m = EDGE_FACTOR * n
    u = torch.zeros(m, dtype=torch.int64, device="cuda")
    v = torch.zeros(m, dtype=torch.int64, device="cuda")
    for _ in range(max(1, (n - 1).bit_length())):
        r = torch.rand(m, device="cuda", generator=gen)
        down = r >= 0.57 + 0.19                                  # quadrants (0.57, 0.19, 0.19, 0.05)
        right = ((r >= 0.57) & ~down) | (r >= 0.57 + 0.19 + 0.19)
        u, v = 2 * u + down, 2 * v + right
    return _csr(n, u % n, v % n)


def _grid(w, h, gen):
    """Lattice with a tenth of its edges deleted (none at vertex 0) and a hundredth of n local shortcuts."""
    n = w * h
    i = torch.arange(n, device="cuda")
    x, y = i % w, torch.div(i, w, rounding_mode="floor")
    a, b = i[x < w - 1], i[y < h - 1]
    u, v = torch.cat([a, b]), torch.cat([a + 1, b + w])
    keep = (torch.rand(u.numel(), device="cuda", generator=gen) >= 0.10) | (u == 0)
    u, v = u[keep], v[keep]
    s = torch.randint(n, (round(0.01 * n),), device="cuda", generator=gen)
    d = torch.randint(-16, 17, (2, s.numel()), device="cuda", generator=gen)
    tx = (x[s] + d[0]).clamp(0, w - 1)
    ty = (y[s] + d[1]).clamp(0, h - 1)
    return _csr(n, torch.cat([u, s]), torch.cat([v, ty * w + tx]))


def _rows(rowptr):
    deg = (rowptr[1:] - rowptr[:-1]).to(torch.int64)
    return torch.repeat_interleave(torch.arange(deg.numel(), device=rowptr.device), deg)


def _weights(n, rowptr, col, wmax, seed):
    """Uniform in [1, wmax], the same on both arcs of an edge: a hash of the pair."""
    u, v = _rows(rowptr), col.to(torch.int64)
    z = torch.minimum(u, v) * n + torch.maximum(u, v) + (seed + 1) * 0x9E3779B1
    for s, c in ((30, 0x3F58476D1CE4E5B9), (27, 0x14D049BB133111EB)):
        z = (z ^ ((z >> s) & ((1 << (64 - s)) - 1))) * c
    return (1 + ((z >> 33) & 0x7FFFFFFF) % wmax).to(torch.int32)


def _graph(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    if case["graph"] == "grid":
        n = case["w"] * case["h"]
        rowptr, col = _grid(case["w"], case["h"], gen)
    else:
        n = case["n"]
        rowptr, col = _rmat(n, gen)
    weighted = case["algo"] in ("sssp", "sssp_batch", "apply")
    wmax = GRID_WMAX if case["graph"] == "grid" else RMAT_WMAX
    return n, rowptr, col, _weights(n, rowptr, col, wmax, seed) if weighted else None


def _sources(case, rowptr, seed):
    """Host int32 array: the hub, the corner (vertex 0), or vertices drawn from those that have arcs."""
    deg = rowptr[1:] - rowptr[:-1]
    where = case.get("source", "random")
    if where == "hub":
        return np.array([int(torch.argmax(deg))], dtype=np.int32)
    if where == "corner":
        return np.zeros(1, dtype=np.int32)
    cand = torch.nonzero(deg > 0).flatten().cpu().numpy()
    rng = np.random.default_rng(seed)
    k = case.get("k", 1)
    return rng.choice(cand, size=k, replace=cand.size < k).astype(np.int32)


def prepare(case, seed):
    n, rowptr, col, w = _graph(case, seed)
    algo = case["algo"]
    s = dict(case, n=n)
    if algo == "new_graph":   # on the host, as a loader leaves it
        s["rowptr"], s["col"] = rowptr.cpu().pin_memory().numpy(), col.cpu().pin_memory().numpy()
        s["rank"] = torch.empty(n, dtype=torch.float32, device="cuda")
        return s
    s["graph_handle"] = g = g2.g2_load_csr(n, rowptr, col, w, symmetric=True)
    rows = (case["k"], n) if algo in ("bfs_batch", "sssp_batch") else (n,)
    if algo in ("bfs", "sssp", "bfs_batch", "sssp_batch", "bc"):
        s["src"] = _sources(case, rowptr, seed)
        s["out"] = torch.empty(rows, dtype=torch.float64 if algo == "bc" else torch.int32, device="cuda")
        s["par"] = torch.empty(n, dtype=torch.int32, device="cuda") if case.get("parent") else None
    elif algo == "cc":
        s["out"] = torch.empty(n, dtype=torch.int32, device="cuda")
    elif algo == "pagerank":
        s["out"] = torch.empty(n, dtype=torch.float32, device="cuda")
    else:   # apply: the frontier's vertices hold distances, the others hold larger ones or none
        rng = np.random.default_rng(seed)
        verts = np.sort(rng.choice(n, size=max(1, int(case["share"] * n)), replace=False)).astype(np.int32)
        dist = rng.integers(200, 600, size=n, dtype=np.int32)
        dist[rng.random(n) < 0.5] = 2**31 - 1
        dist[verts] = rng.integers(0, 400, size=verts.size, dtype=np.int32)
        s["dist0"] = torch.from_numpy(dist).cuda()
        s["out"] = torch.empty_like(s["dist0"])
        s["fin"], s["fout"] = (g2.g2_frontier_create(g, g2.G2_FRONTIER_SPARSE) for _ in range(2))
        s["fin"].set(verts)
        s["sched"] = g2.schedule(case["lb"])
    return s


def run(s):
    algo = s["algo"]
    if algo == "new_graph":
        g = g2.g2_load_csr(s["n"], s["rowptr"], s["col"], symmetric=True, prepare_pagerank=True)
        g2.g2_pagerank(g, DAMPING, ROUNDS, s["rank"])
        g.free()
        return s["rank"]
    g, out = s["graph_handle"], s["out"]
    if algo == "bfs":
        g2.g2_bfs(g, int(s["src"][0]), out, s["par"])
        return out if s["par"] is None else (out, s["par"])
    if algo == "cc":
        g2.g2_cc(g, out)
    elif algo == "pagerank":
        g2.g2_pagerank(g, DAMPING, ROUNDS, out)
    elif algo == "sssp":
        g2.g2_sssp_delta(g, int(s["src"][0]), s["delta"], out)
    elif algo == "bfs_batch":
        g2.g2_bfs_batch(g, s["src"], out)
    elif algo == "sssp_batch":
        g2.g2_sssp_batch(g, s["src"], s["delta"], out)
    elif algo == "bc":
        g2.g2_bc(g, s["src"], out)
    else:
        out.copy_(s["dist0"])
        return out, g2.g2_edgeset_apply(g, g2.G2_OP_RELAX_MIN, s["fin"], out, None, s["sched"], s["fout"])
    return out


# ------------------------------------------------------------------------------------------- work, exact
def _size(case):
    """(n, expected arcs): RMAT's share of duplicate samples shrinks by 0.836 a scale from 0.186 at scale 14."""
    if case["graph"] == "grid":
        n = case["w"] * case["h"]
        return n, int(2 * (0.9 * (2 * n - case["w"] - case["h"]) + 0.01 * n))
    n = case["n"]
    return n, int(2 * EDGE_FACTOR * n * (1 - min(0.5, 0.1864 * 0.836 ** (math.log2(n) - 14))))


def work(case):
    """Bytes: row offsets, arcs (ids, and weights where the call takes them) and outputs once.  A BFS or a component
    labelling does not need every arc: one per vertex (the one that reaches it).  Operations: one a relaxed arc."""
    n, m = _size(case)
    algo = case["algo"]
    if algo == "bfs":
        return {"bytes": 4 * n + 4 * n + 4 * n * (2 if case["parent"] else 1), "flops": n}
    if algo == "cc":
        return {"bytes": 4 * n + 4 * n + 4 * n, "flops": n}
    if algo == "bfs_batch":
        return {"bytes": 4 * n + 4 * m + 4 * n * case["k"], "flops": m}
    if algo in ("sssp", "sssp_batch"):
        k = case.get("k", 1)
        return {"bytes": 4 * n + 8 * m + 4 * n * k, "flops": m * k}
    if algo == "bc":
        return {"bytes": 4 * n + 4 * m + 8 * n, "flops": 2 * m * case["k"]}
    if algo == "apply":
        arcs = m * case["share"]
        return {"bytes": int(8 * n * case["share"] + 8 * arcs + 8 * n), "flops": int(arcs)}
    # PageRank: every round needs every arc, but the layout may stay on the chip between rounds only in part
    return {"bytes": ROUNDS * (4 * m + 8 * n), "flops": ROUNDS * m}


def _exact_pagerank(n, rowptr, col):
    deg = (rowptr[1:] - rowptr[:-1]).double()
    rows, c = _rows(rowptr), col.to(torch.int64)
    x = torch.full((n,), 1.0 / n, dtype=torch.float64, device="cuda")
    for _ in range(ROUNDS):
        share = torch.where(deg > 0, x / deg.clamp(min=1), torch.zeros_like(x))
        lost = x[deg == 0].sum()
        y = torch.zeros_like(x).index_add_(0, rows, share[c])
        x = (1 - DAMPING) / n + DAMPING * (y + lost / n)
    return x


def _exact_bc(n, rowptr, col, srcs):
    rows, c = _rows(rowptr), col.to(torch.int64)
    bc = torch.zeros(n, dtype=torch.float64, device="cuda")
    for src in srcs:
        depth = torch.full((n,), -1, dtype=torch.int64, device="cuda")
        depth[int(src)] = 0
        d = 0
        while True:
            reach = torch.zeros(n, dtype=torch.bool, device="cuda")
            reach[c[depth[rows] == d]] = True
            reach &= depth < 0
            if not bool(reach.any()):
                break
            d += 1
            depth[reach] = d
        du = depth[rows]
        on = (du >= 0) & (depth[c] == du + 1)               # arcs of shortest paths, by level
        u, v, lev = rows[on], c[on], du[on]
        order = torch.argsort(lev)
        u, v = u[order], v[order]
        ends = torch.cumsum(torch.bincount(lev, minlength=d), 0).tolist()
        level = [slice(a, b) for a, b in zip([0] + ends, ends)]
        sigma = torch.zeros(n, dtype=torch.float64, device="cuda")
        sigma[int(src)] = 1
        for t in level:
            sigma.index_add_(0, v[t], sigma[u[t]])
        delta = torch.zeros_like(sigma)
        for t in reversed(level):
            delta.index_add_(0, u[t], sigma[u[t]] / sigma[v[t]] * (1 + delta[v[t]]))
        delta[int(src)] = 0
        bc += delta
    return bc


def exact(case, seed):
    algo = case["algo"]
    if algo not in ("pagerank", "new_graph", "bc"):
        return None                                          # whole numbers
    if algo == "bc" and case["graph"] == "grid" and case["w"] + case["h"] > 600:
        return None                                          # path counts near the end of the 64-bit range
    n, rowptr, col, _ = _graph(case, seed)
    if algo == "bc":
        return _exact_bc(n, rowptr, col, _sources(case, rowptr, seed))
    return _exact_pagerank(n, rowptr, col)
