"""The work that users of this library have it do, as timed cases.

A case is one call (or a call and what follows from it) through the Python
binding on one seeded graph or batch of graphs:

  call     count       tc_count: T from device arrays
           vertex      tc_count_per_vertex: T, t[n], deg[n]
           cluster     tc_count_per_vertex, then tc_clustering: cc[n] and the
                       transitivity ratio as well
           host        tc_count_host: T from page-locked host arrays
           workspace   tc_count_ws: T in a workspace that the caller keeps
           batch       tc_count_batch: T of every graph of a batch
           engine      Engine.count: the same through a persistent engine
  graph    er          uniform distinct edges
           rmat        R-MAT (a, b, c = .57, .19, .19), permuted ids, distinct edges
           rmat_raw    the same, self-loops and repeats left in the input
           ba          preferential attachment, k edges per new vertex
           ws          ring of k neighbours on either side, a tenth rewired
           rgg         random geometric graph of a given mean degree
           mixed       a batch: even graphs er, odd ones R-MAT, sizes
                       log-uniform, mean degree uniform
  both     every edge given in both directions (the paper's input format)

The graphs are made on the GPU with torch, from the seed alone.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1503_00576_gb300 as tc

RMAT = (0.57, 0.19, 0.19)
MOST_WEDGES = 1_500_000_000  # exact() enumerates no more forward wedges than these


def listed():
    return [
        # one small graph, counted on its own: launches and latency
        {"name": "er1k_count", "call": "count", "graph": "er", "n": 1003, "m": 8191},
        # the smallest workload of the benchmark, with the clustering
        # coefficients that triangles are counted for
        {"name": "er16k_cluster", "call": "cluster", "graph": "er", "n": 16384, "m": 131072},
        # the smallest Kronecker graph of the paper's Table 1
        {"name": "kron16_count", "call": "count", "graph": "rmat", "n": 1 << 16, "m": 2_500_000},
        # Table 1's Kronecker 18, timed as the paper does: from host memory
        {"name": "kron18_host", "call": "host", "graph": "rmat", "n": 1 << 18, "m": 10_500_000},
        # raw generator output, self-loops and repeats for the library to drop
        {"name": "rmat20_vertex", "call": "vertex", "graph": "rmat_raw", "n": 1 << 20,
         "m": 16 << 20},
        # Table 1's Barabasi-Albert network: few triangles, lists of equal length
        {"name": "ba200k_count", "call": "count", "graph": "ba", "n": 200_000, "k": 50},
        # Table 1's Watts-Strogatz network in the paper's format, in a loop
        # that keeps its workspace
        {"name": "ws1m_both_ws", "call": "workspace", "graph": "ws", "n": 1_000_000, "k": 25,
         "both": True},
        # high clustering and short lists: preprocessing outweighs counting
        {"name": "rgg4m_cluster", "call": "cluster", "graph": "rgg", "n": 1 << 22,
         "degree": 32.0},
        # Table 1's largest Kronecker graph
        {"name": "kron21_count", "call": "count", "graph": "rmat", "n": 1 << 21,
         "m": 91_000_000},
        # the benchmark's main workload
        {"name": "rmat24_vertex", "call": "vertex", "graph": "rmat", "n": 1 << 24,
         "m": 180_000_000},
        # a part of the benchmark's batch of 4096 graphs
        {"name": "batch64", "call": "batch", "graph": "mixed", "graphs": 64, "log2_lo": 8.0,
         "log2_hi": 18.0, "deg_lo": 4.0, "deg_hi": 64.0, "sizes": 7},
        # what a serving loop hands its engine: many small graphs, the engine
        # sized above them
        {"name": "engine300_small", "call": "engine", "graph": "mixed", "graphs": 300,
         "log2_lo": 8.0, "log2_hi": 12.0, "deg_lo": 4.0, "deg_hi": 32.0, "sizes": 11},
    ]


def _between(rng, lo, hi):
    """An integer, uniform over its logarithm, odd as often as not."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["count", "count", "vertex", "vertex", "cluster", "host", "workspace",
                       "batch", "engine"])
    if call in ("batch", "engine"):
        lo = rng.uniform(8.0, 11.0)
        return {"call": call, "graph": "mixed", "graphs": _between(rng, 2, 200), "log2_lo": lo,
                "log2_hi": lo + rng.uniform(1.0, 5.0), "deg_lo": 4.0,
                "deg_hi": rng.uniform(8.0, 64.0), "sizes": rng.randrange(1 << 20)}
    graph = rng.choice(["er", "rmat", "rmat", "rmat_raw", "ba", "ws", "rgg"])
    n = _between(rng, 500, 4_000_000)
    if graph in ("er", "rmat", "rmat_raw"):
        # mean degrees of 8 to 80, as from the benchmark's to Table 1's
        m = min(int(n * rng.uniform(4.0, 40.0)), 60_000_000, n * (n - 1) // 16)
        if graph != "er":  # a generator's scale
            n = 1 << max(9, round(math.log2(n)))
            m = min(m, n * n // 64)
        case = {"call": call, "graph": graph, "n": n, "m": m}
    elif graph in ("ba", "ws"):
        n = min(n, 1_000_000)
        case = {"call": call, "graph": graph, "n": n, "k": rng.randrange(3, 50)}
    else:
        case = {"call": call, "graph": graph, "n": n, "degree": rng.uniform(6.0, 40.0)}
    if rng.random() < 0.25:
        case["both"] = True
    return case


# ---------------------------------------------------------------------------
# graphs
# ---------------------------------------------------------------------------
def _rand(g, m):
    return torch.rand(m, device="cuda", generator=g)


def _randint(g, hi, m):
    return torch.randint(hi, (m,), device="cuda", generator=g)


def _rmat_ids(g, bits, m):
    """m draws of two `bits`-bit ids (int64), before any permutation."""
    a, b, c = RMAT
    u = torch.zeros(m, dtype=torch.int64, device="cuda")
    v = torch.zeros_like(u)
    for _ in range(bits):
        r = _rand(g, m)
        low = r >= a + b  # the lower half of the matrix
        u.mul_(2).add_(low)
        v.mul_(2).add_(((r >= a) & ~low) | (r >= a + b + c))
    return u, v


def _distinct(g, u, v, n, m=None):
    """The distinct edges among the pairs, without loops, in random order and
    direction; m of them if given (None if there are fewer)."""
    keep = u != v
    u, v = u[keep], v[keep]
    key = torch.unique(torch.minimum(u, v) * n + torch.maximum(u, v))
    if m is not None and key.numel() < m:
        return None
    key = key[torch.randperm(key.numel(), device="cuda", generator=g)[:m]]
    return _direct(g, key // n, key % n)


def _direct(g, u, v):
    flip = _rand(g, u.numel()) < 0.5
    return torch.where(flip, v, u), torch.where(flip, u, v)


def _shuffle(g, u, v, n):
    """Permuted ids, random order and direction."""
    ids = torch.randperm(n, device="cuda", generator=g)
    order = torch.randperm(u.numel(), device="cuda", generator=g)
    return _direct(g, ids[u[order]], ids[v[order]])


def _er(g, n, m):
    draws = m + m // 8 + 64
    while True:
        pairs = _distinct(g, _randint(g, n, draws), _randint(g, n, draws), n, m)
        if pairs is not None:
            return pairs
        draws += draws // 2


def _rmat(g, n, m, raw):
    bits = n.bit_length() - 1
    ids = torch.randperm(n, device="cuda", generator=g)
    draws = m if raw else m + m // 8 + 64
    while True:
        u, v = _rmat_ids(g, bits, draws)
        u, v = ids[u], ids[v]
        if raw:
            return u, v
        pairs = _distinct(g, u, v, n, m)
        if pairs is not None:
            return pairs
        del u, v
        draws += draws // 2


def _ba(g, n, k):
    """A clique on k + 1 vertices; every later vertex joins k ends drawn from
    all edge ends so far (repeats dropped, about one edge in a hundred)."""
    k = min(k, n - 1)
    seed = torch.triu_indices(k + 1, k + 1, 1, device="cuda")
    s = seed.shape[1]
    new = torch.arange(k + 1, n, device="cuda").repeat_interleave(k)
    # edge ends: slot 2e the new vertex of edge e, slot 2e + 1 what it joins,
    # a uniform slot below its vertex's first edge
    before = 2 * (s + (new - (k + 1)) * k)
    at = (torch.rand(new.numel(), device="cuda", generator=g, dtype=torch.float64)
          * before).long()
    while True:  # a slot that was drawn itself stands for the slot it drew
        drawn = (at >= 2 * s) & (at % 2 == 1)
        if not bool(drawn.any()):
            break
        at = torch.where(drawn, at[((at - 2 * s) // 2).clamp_(min=0)], at)
    first = torch.cat([seed[0], new])
    to = torch.where(at % 2 == 0, first[at // 2], seed[1][(at // 2).clamp(max=s - 1)])
    ids = torch.randperm(n, device="cuda", generator=g)
    return _distinct(g, ids[first], ids[torch.cat([seed[1], to])], n)


def _ws(g, n, k):
    k = min(k, (n - 2) // 4)
    u = torch.arange(n, device="cuda").repeat_interleave(k)
    near = torch.arange(1, k + 1, device="cuda").repeat(n)
    far = k + 1 + _randint(g, n - 2 * k - 1, n * k)
    return _shuffle(g, u, (u + torch.where(_rand(g, n * k) < 0.1, far, near)) % n, n)


def _rgg(g, n, degree):
    r = min(math.sqrt(degree / (math.pi * n)), 0.5)
    side = int(1.0 / r)
    xy = torch.rand(2, n, device="cuda", generator=g, dtype=torch.float64)
    cell = (xy[1] * side).long() * side + (xy[0] * side).long()
    cell, order = torch.sort(cell, stable=True)
    x, y = xy[0][order], xy[1][order]
    start = torch.searchsorted(cell, torch.arange(side * side + 1, device="cuda"))
    cx, cy = cell % side, cell // side
    us, vs = [], []
    for dx, dy in ((0, 0), (1, 0), (-1, 1), (0, 1), (1, 1)):
        ok = (cx + dx >= 0) & (cx + dx < side) & (cy + dy < side)
        c = torch.where(ok, cell + dy * side + dx, cell)
        lo, hi = start[c], start[c + 1]
        if (dx, dy) == (0, 0):
            lo = torch.arange(1, n + 1, device="cuda")
        count = torch.where(ok, hi - lo, 0)
        u = torch.arange(n, device="cuda").repeat_interleave(count)
        at = torch.arange(u.numel(), device="cuda") - (count.cumsum(0) - count)[u]
        v = lo[u] + at
        close = (x[u] - x[v]) ** 2 + (y[u] - y[v]) ** 2 < r * r
        us.append(u[close])
        vs.append(v[close])
    return _shuffle(g, torch.cat(us), torch.cat(vs), n)


def _mixed_sizes(case):
    """(n, m) of the graphs of a batch: part of the case, not of the seed."""
    rng = np.random.default_rng(case["sizes"])
    count = case["graphs"]
    lo, hi = case["log2_lo"], case["log2_hi"]
    n = np.floor(np.exp2(lo + (hi - lo) * rng.random(count))).astype(np.int64)
    d = case["deg_lo"] + (case["deg_hi"] - case["deg_lo"]) * rng.random(count)
    return n, np.minimum(np.floor(n * d / 2).astype(np.int64), n * (n - 1) // 4)


def _mixed(g, case):
    """The graphs of a batch back to back, with their pairs' and vertices'
    counts (R-MAT graphs of any n: ids are fractions of n; repeats dropped, so
    a graph may have a few pairs fewer than its size says)."""
    n, m = _mixed_sizes(case)
    nd, md = torch.from_numpy(n).cuda(), torch.from_numpy(m).cuda()
    graph = torch.arange(len(n), device="cuda").repeat_interleave(md)
    total = graph.numel()
    ru, rv = _rmat_ids(g, 20, total)
    rmat = graph % 2 == 1
    fu = torch.where(rmat, ru / 2.0 ** 20, torch.rand(total, device="cuda", generator=g,
                                                      dtype=torch.float64))
    fv = torch.where(rmat, rv / 2.0 ** 20, torch.rand(total, device="cuda", generator=g,
                                                      dtype=torch.float64))
    nv = nd[graph]
    u, v = (fu * nv).long(), (fv * nv).long()
    keep = u != v
    graph, u, v = graph[keep], u[keep], v[keep]
    key = torch.unique((graph << 40) | (torch.minimum(u, v) << 20) | torch.maximum(u, v))
    key = key[torch.randperm(key.numel(), device="cuda", generator=g)]
    key = key[torch.sort(key >> 40, stable=True).indices]
    counts = torch.bincount(key >> 40, minlength=len(n)).cpu().numpy()
    u, v = _direct(g, (key >> 20) & 0xFFFFF, key & 0xFFFFF)
    offsets = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    return u, v, offsets, n.astype(np.int32)


def _pairs(case, seed):
    """(src, dst) of a case's graph as int32 CUDA tensors."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    n, kind = case["n"], case["graph"]
    if kind == "er":
        u, v = _er(g, n, case["m"])
    elif kind in ("rmat", "rmat_raw"):
        u, v = _rmat(g, n, case["m"], kind == "rmat_raw")
    elif kind == "ba":
        u, v = _ba(g, n, case["k"])
    elif kind == "ws":
        u, v = _ws(g, n, case["k"])
    else:
        u, v = _rgg(g, n, case["degree"])
    if case.get("both"):
        order = torch.randperm(2 * u.numel(), device="cuda", generator=g)
        u, v = torch.cat([u, v])[order], torch.cat([v, u])[order]
    return u.int(), v.int()


def prepare(case, seed):
    state = {"call": case["call"]}
    if case["graph"] == "mixed":
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        u, v, state["offsets"], state["vertices"] = _mixed(g, case)
        state["src"], state["dst"] = u.int(), v.int()
        del u, v
        if case["call"] == "engine":
            n, m = _mixed_sizes(case)
            # what a serving loop sets aside: a quarter more than its batches hold
            state["engine"] = tc.Engine(int(m.sum() * 5 // 4), int(n.sum() * 5 // 4),
                                        2 * case["graphs"])
    else:
        src, dst = _pairs(case, seed)
        state["n"] = case["n"]
        if case["call"] == "host":
            src, dst = src.cpu().pin_memory(), dst.cpu().pin_memory()
        elif case["call"] == "workspace":
            state["ws"] = torch.empty(tc.tc_workspace_bytes(src.numel(), case["n"]),
                                      dtype=torch.uint8, device="cuda")
        state["src"], state["dst"] = src, dst
    torch.cuda.empty_cache()  # the generators' scratch; the library does not allocate from torch
    return state


def run(state):
    call, src, dst = state["call"], state["src"], state["dst"]
    if call == "count":
        return tc.tc_count(src, dst, state["n"])
    if call == "vertex":
        return tc.tc_count_per_vertex(src, dst, state["n"])
    if call == "cluster":
        total, t, deg = tc.tc_count_per_vertex(src, dst, state["n"])
        cc, transitivity = tc.tc_clustering(t, deg)
        return total, t, deg, cc, transitivity
    if call == "host":
        return tc.tc_count_host(src, dst, state["n"])
    if call == "workspace":
        return tc.tc_count_ws(src, dst, state["n"], state["ws"])
    if call == "batch":
        return tc.tc_count_batch(src, dst, state["offsets"], state["vertices"])
    return state["engine"].count(src, dst, state["offsets"], state["vertices"])


def _pair_count(case):
    """Pairs of a case's input (an expectation where the graph is random)."""
    n, kind = case.get("n"), case["graph"]
    if kind == "mixed":
        return int(_mixed_sizes(case)[1].sum())
    if kind == "ba":
        k = min(case["k"], n - 1)
        m = k * (k + 1) // 2 + (n - k - 1) * k
    elif kind == "ws":
        m = n * min(case["k"], (n - 2) // 4)
    elif kind == "rgg":
        m = int(n * min(case["degree"], n / 2) / 2)
    else:
        m = case["m"]
    return 2 * m if case.get("both") else m


def work(case):
    """Every pair read once, every result written once.  The comparisons that
    intersections need depend on the graph and are not counted."""
    out = 8 * case["graphs"] if case["graph"] == "mixed" else 8
    if case["call"] in ("vertex", "cluster"):
        out += 12 * case["n"]  # t int64, deg int32
    if case["call"] == "cluster":
        out += 8 * case["n"] + 8  # cc float64
    return {"bytes": 8 * _pair_count(case) + out, "flops": 0}


# ---------------------------------------------------------------------------
# exact values
# ---------------------------------------------------------------------------
def _exact_graph(u, v, n):
    """(T, t, deg) by enumerating the wedges of the forward lists; None where
    there are too many."""
    u, v = u.long(), v.long()
    keep = u != v
    key = torch.unique(torch.minimum(u[keep], v[keep]) * n + torch.maximum(u[keep], v[keep]))
    a, b = key // n, key % n
    deg = torch.bincount(torch.cat([a, b]), minlength=n)
    rank = torch.empty(n, dtype=torch.int64, device="cuda")
    rank[torch.sort(deg, stable=True).indices] = torch.arange(n, device="cuda")
    key = torch.sort(torch.minimum(rank[a], rank[b]) * n + torch.maximum(rank[a], rank[b])).values
    a, b = key // n, key % n
    end = torch.cumsum(torch.bincount(a, minlength=n), 0)[a]
    later = end - 1 - torch.arange(key.numel(), device="cuda")  # entries after b in a's list
    cum = torch.cumsum(later, 0)
    if key.numel() == 0 or int(cum[-1]) > MOST_WEDGES:
        return None
    t = torch.zeros(n, dtype=torch.int64, device="cuda")
    step, e0 = 1 << 26, 0
    while e0 < key.numel():
        base = int(cum[e0 - 1]) if e0 else 0
        e1 = max(e0 + 1, int(torch.searchsorted(cum, base + step)))
        e = torch.arange(e0, e1, device="cuda").repeat_interleave(later[e0:e1])
        at = torch.arange(e.numel(), device="cuda") - (cum[e] - later[e] - base)
        w = b[e + 1 + at]
        find = b[e] * n + w
        hit = key[torch.searchsorted(key, find).clamp_(max=key.numel() - 1)] == find
        e, w = e[hit], w[hit]
        t += torch.bincount(torch.cat([a[e], b[e], w]), minlength=n)
        e0 = e1
    return int(t.sum()) // 3, t[rank], deg


def exact(case, seed):
    """T, t and deg by enumeration, cc and transitivity from them in float64."""
    if case["graph"] == "mixed" or case["call"] != "cluster":
        return None  # whole numbers alone
    src, dst = _pairs(case, seed)
    found = _exact_graph(src, dst, case["n"])
    if found is None:
        return None
    total, t, deg = found
    open_or_closed = deg * (deg - 1)
    cc = torch.where(open_or_closed > 0, 2.0 * t.double() / open_or_closed.clamp(min=1).double(),
                     torch.zeros((), dtype=torch.float64, device="cuda"))
    wedges = int((open_or_closed // 2).sum())
    return total, t, deg.int(), cc, 3.0 * total / wedges if wedges else 0.0
