"""The work a program gives this library, as cases that can be timed.

A case names a call (`call`), the graph it is made on and its sizes.  The
graphs are the families of the repository's own workloads, drawn on the
device from the seed: R-MAT with (a, b, c, d) = (.57, .19, .19, .05)
and a random vertex permutation, a 4-neighbour grid with diagonals and a
Chung-Lu overlay, and sets of small Barabasi-Albert and planted-hierarchy
graphs.  A case fixes the vertices and the distinct edges of its graphs, so
that results have the same shapes for every seed: the random pairs of a
graph are drawn until that many distinct edges are there (`pairs` is what
this takes, within a hundredth or so).  Calls:

  full      triangle_centrality(): pair list in, all results out
  recount   count and centrality again on a Graph that is kept
  edges     per-edge triangle counts on a Graph that is kept
  batch     a set of small graphs, built, run and released
  rerun     a kept Batch, run again
  noalloc   counts and centrality of a small CSR without any allocation
  serve     requests of host pairs through a Server, host results back
"""
import math

import numpy as np
import torch

import paper_2105_00110_gb300 as tc

ABC = (0.57, 0.19, 0.19)          # R-MAT quadrants of the repository's workloads
MAX_EXACT_WEDGES = 3 * 10**9      # what exact() lists within seconds


def listed():
    return [
        # the smallest configuration: one small graph, where launches and host work count
        {"name": "full-rmat-12", "call": "full", "graph": "rmat", "pairs": 65536, "ids": 32},
        # an analysis of an ordinary social graph kept as 64-bit ids, an odd number of pairs
        {"name": "full-rmat-16-i64", "call": "full", "graph": "rmat", "pairs": 1000003, "ids": 64},
        # a graph of sixteen million pairs
        {"name": "full-rmat-20", "call": "full", "graph": "rmat", "pairs": 1 << 24, "ids": 32},
        # the headline configuration
        {"name": "full-rmat-24", "call": "full", "graph": "rmat", "pairs": 1 << 28, "ids": 32},
        # a mesh-like graph of a million vertices with a few hubs, odd side, 64-bit ids
        {"name": "full-grid-999-i64", "call": "full", "graph": "grid", "side": 999, "ids": 64},
        # the grid configuration
        {"name": "full-grid-4096", "call": "full", "graph": "grid", "side": 4096, "ids": 32},
        # a graph kept by the program, counted again
        {"name": "recount-rmat-22", "call": "recount", "graph": "rmat", "pairs": 1 << 26, "ids": 32},
        # per-edge counts (truss-style filtering) on a kept graph, a ragged number of pairs
        {"name": "edges-rmat-20", "call": "edges", "graph": "rmat", "pairs": 12345677, "ids": 32},
        # the batched configuration, from pair lists to results
        {"name": "batch-8192", "call": "batch", "graph": "set", "count": 8192, "n_max": 65536},
        # a smaller set of small graphs, kept and run again
        {"name": "rerun-500", "call": "rerun", "graph": "set", "count": 500, "n_max": 20000},
        # a small graph inside a loop that must not allocate
        {"name": "noalloc-rmat-12", "call": "noalloc", "graph": "rmat", "pairs": 65536, "ids": 32},
        # a burst of requests of all sizes at a server
        {"name": "serve-24", "call": "serve", "graph": "burst", "count": 24, "pairs_max": 10000000},
    ]


def _log_between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["full", "full", "full", "recount", "edges", "batch", "rerun", "noalloc", "serve"])
    if call == "noalloc":
        return {"call": call, "graph": "rmat", "pairs": _log_between(rng, 300, 900000), "ids": 32}
    if call in ("batch", "rerun"):
        return {"call": call, "graph": "set", "count": _log_between(rng, 16, 5000),
                "n_max": _log_between(rng, 1000, 65536)}
    if call == "serve":
        return {"call": call, "graph": "burst", "count": rng.randint(4, 28),
                "pairs_max": _log_between(rng, 30000, 10000000)}
    ids = rng.choice([32, 32, 64])
    if rng.random() < 0.3:
        return {"call": call, "graph": "grid", "side": _log_between(rng, 32, 4000), "ids": ids}
    return {"call": call, "graph": "rmat", "pairs": _log_between(rng, 4000, 100000000), "ids": ids}


# ------------------------------------------------------------------ graphs
def _scale(pairs):
    return max(4, math.ceil(math.log2(pairs / 16)))


def _until(src, dst, n, edges):
    """The pairs up to the one that brings the `edges`-th distinct edge."""
    lo, hi = torch.minimum(src, dst).long(), torch.maximum(src, dst).long()
    key, at = torch.sort(torch.where(lo == hi, n * n, lo * n + hi), stable=True)
    new = torch.ones(len(key), dtype=torch.bool, device="cuda")
    new[1:] = key[1:] != key[:-1]
    first = torch.sort(at[new & (key < n * n)]).values
    if len(first) < edges:
        raise RuntimeError("%d distinct edges drawn, %d wanted" % (len(first), edges))
    end = int(first[edges - 1]) + 1
    return src[:end].clone(), dst[:end].clone(), n


def _rmat(pairs, gen):
    """R-MAT pairs over 2^scale vertices, permuted labels."""
    scale = _scale(pairs)
    n = 1 << scale
    a, b, c = ABC
    src = torch.zeros(pairs, dtype=torch.int32, device="cuda")
    dst = torch.zeros(pairs, dtype=torch.int32, device="cuda")
    for _ in range(scale):
        x = torch.rand(pairs, device="cuda", generator=gen)
        s = x >= a + b                       # quadrants c, d
        d = ((x >= a) & ~s) | (x >= a + b + c)   # quadrants b, d
        src.mul_(2).add_(s)
        dst.mul_(2).add_(d)
    perm = torch.randperm(n, device="cuda", generator=gen, dtype=torch.int32)
    return _until(perm[src], perm[dst], n, _rmat_edges(pairs))


def _grid_edges(side):
    return int(side * side * (3.78 - 3.0 / side))


def _grid(side, gen):
    """side x side grid, a diagonal per cell with probability 0.05, and a
    Chung-Lu overlay (exponent 2.1, mean degree about 4) on permuted vertices."""
    n = side * side
    ids = torch.arange(n, device="cuda").view(side, side)
    cell = torch.rand(side - 1, side - 1, device="cuda", generator=gen) < 0.05
    perm = torch.randperm(n, device="cuda", generator=gen)
    # vertex k with weight (k + 1)^(-1 / 1.1), by the inverse of the weights' integral
    x = torch.rand(2, 23 * n // 10, device="cuda", dtype=torch.float64, generator=gen)
    ends = perm[((1 + x * ((n + 1) ** (1 / 11) - 1)).pow(11) - 1).long().clamp_(0, n - 1)]
    src = torch.cat([ids[:, :-1].reshape(-1), ids[:-1].reshape(-1), ids[:-1, :-1][cell], ends[0]])
    dst = torch.cat([ids[:, 1:].reshape(-1), ids[1:].reshape(-1), ids[1:, 1:][cell], ends[1]])
    return _until(src, dst, n, _grid_edges(side))


def _triangular(j):
    """(a, b), a < b, of the j-th pair (b major)."""
    b = ((1 + (1 + 8 * j).double().sqrt()) / 2).long()
    b -= (b * (b - 1) // 2 > j).long()
    return j - b * (b - 1) // 2, b


def _spread(counts):
    """For counts[k] elements of group k: the group and the place in it of each."""
    k = torch.repeat_interleave(torch.arange(len(counts), device="cuda"), counts)
    first = counts.cumsum(0) - counts
    return k, torch.arange(len(k), device="cuda") - first[k]


def _below(bound, gen):
    """Uniform whole numbers in [0, bound) for a tensor of bounds."""
    x = torch.rand(bound.shape, device="cuda", dtype=torch.float64, generator=gen)
    return torch.minimum((x * bound).long(), bound - 1)


def _graph_set(count, n_max, gen):
    """Pairs (local ids), pair offsets and vertex counts of `count` graphs, n
    log-uniform in [32, n_max]: half Barabasi-Albert (2 to 8 edges a vertex),
    half hierarchies (a root, 4 to 32 cliques of 3 to 12, leaves on the
    clique members, one noise edge for a hundredth of the vertices).  The
    sizes belong to the case, the edges to the seed; a repeated edge is
    drawn again."""
    rng = np.random.default_rng([count, n_max])
    n = np.rint(np.exp(rng.uniform(math.log(32), math.log(n_max), count))).astype(np.int64)
    ba = rng.random(count) < 0.5
    mm = rng.integers(2, 9, count)
    c, k = rng.integers(4, 33, count), rng.integers(3, 13, count)
    n = np.where(ba, np.maximum(n, mm + 1), np.maximum(n, 1 + c * k))
    gn, gmm, gc, gk = (torch.from_numpy(x).cuda() for x in (n, mm, c, k))
    is_ba = torch.from_numpy(ba).cuda()

    # Barabasi-Albert: edge j of a graph joins its vertex to an earlier edge's end
    seed_edges = gmm * (gmm + 1) // 2
    ne = torch.where(is_ba, seed_edges + (gn - gmm - 1) * gmm, 0)
    g1, j = _spread(ne)
    lead = seed_edges[g1]
    grown = j >= lead
    ca, cb = _triangular(torch.minimum(j, lead - 1))
    v = gmm[g1] + 1 + (j - lead) // gmm[g1]
    u1 = torch.where(grown, v, ca)
    first = (ne.cumsum(0) - ne)[g1]
    slot = _below(torch.where(grown, 2 * (lead + (v - gmm[g1] - 1) * gmm[g1]), 1), gen) + 2 * first
    # slot 2e is edge e's first end, 2e + 1 its second: follow second ends of
    # grown edges until the slot names a vertex
    while True:
        open_ = grown & (slot % 2 == 1) & grown[slot // 2]
        if not bool(open_.any()):
            break
        slot = torch.where(open_, slot[slot // 2], slot)
    v1 = torch.where(grown, torch.where(slot % 2 == 0, u1[slot // 2], cb[slot // 2]), cb)
    del v, lead, first

    # hierarchies
    zero = torch.zeros_like(gn)
    g2, q = _spread(torch.where(is_ba, zero, gc))
    u2, v2 = torch.zeros_like(q), 1 + q * gk[g2] + _below(gk[g2], gen)
    per = gk * (gk - 1) // 2
    g3, j = _spread(torch.where(is_ba, zero, gc * per))
    ca, cb = _triangular(j % per[g3])
    at = 1 + j // per[g3] * gk[g3]
    u3, v3 = at + ca, at + cb
    g4, j = _spread(torch.where(is_ba, zero, gn - 1 - gc * gk))
    u4, v4 = 1 + gc[g4] * gk[g4] + j, 1 + _below(gc[g4] * gk[g4], gen)
    g5, _ = _spread(torch.where(is_ba, zero, (gn + 99) // 100))
    u5, v5 = _below(gn[g5], gen), _below(gn[g5], gen)

    g = torch.cat([g1, g2, g3, g4, g5])
    u, v = torch.cat([u1, u2, u3, u4, u5]), torch.cat([v1, v2, v3, v4, v5])
    del g1, g2, g3, g4, g5, u1, u2, u3, u4, u5, v1, v2, v3, v4, v5, ca, cb, at, j, q, slot, open_, grown
    start, total = gn.cumsum(0) - gn, int(gn.sum())
    while True:
        key, at = torch.sort((start[g] + torch.minimum(u, v)) * total + start[g] + torch.maximum(u, v), stable=True)
        again = torch.cat([at[1:][key[1:] == key[:-1]], (u == v).nonzero()[:, 0]])
        if not len(again):
            break
        v[again] = _below(gn[g[again]], gen)
    order = torch.sort(g.to(torch.int32), stable=True).indices
    src, dst = u.to(torch.int32)[order], v.to(torch.int32)[order]
    off = np.zeros(count + 1, np.int64)
    off[1:] = torch.bincount(g, minlength=count).cumsum(0).cpu().numpy()
    return src, dst, off, n


def _burst(case, gen):
    """A burst's requests: R-MAT graphs, pair counts stratified over the
    logarithm of [1000, pairs_max]."""
    count = case["count"]
    rng = np.random.default_rng([count, case["pairs_max"]])
    at = (np.arange(count) + rng.random(count)) / count
    sizes = [int(round(1000 * (case["pairs_max"] / 1000) ** x)) for x in rng.permutation(at)]
    return [_rmat(p, gen) for p in sizes]


def _pairs(case, gen):
    src, dst, n = _rmat(case["pairs"], gen) if case["graph"] == "rmat" else _grid(case["side"], gen)
    dt = torch.int32 if case["ids"] == 32 else torch.int64
    return src.to(dt), dst.to(dt), n


def _distinct(src, dst, n):
    """The simple graph's edges (u < v), sorted."""
    lo, hi = torch.minimum(src, dst).long(), torch.maximum(src, dst).long()
    key = torch.unique((lo * n + hi)[lo != hi])
    return key // n, key % n


def _csr(src, dst, n):
    u, v = _distinct(src, dst, n)
    key = torch.sort(torch.cat([u * n + v, v * n + u])).values
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.bincount(key // n, minlength=n).cumsum(0)
    return row_ptr, (key % n).to(torch.int32)


def _pinned(t, dtype):
    out = torch.empty(t.shape, dtype=dtype, pin_memory=True)
    out.copy_(t)
    return out


def _inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if case["graph"] == "set":
        return _graph_set(case["count"], case["n_max"], gen)
    if case["graph"] == "burst":
        return _burst(case, gen)
    return _pairs(case, gen)


# --------------------------------------------------------------- the calls
def prepare(case, seed):
    call = case["call"]
    x = _inputs(case, seed)
    if call == "full":
        return {"call": call, "src": x[0], "dst": x[1], "n": x[2]}
    if call in ("recount", "edges"):
        return {"call": call, "graph": tc.Graph(x[0], x[1], x[2])}
    if call == "batch":
        return {"call": call, "set": x}
    if call == "rerun":
        return {"call": call, "batch": tc.Batch(*x)}
    if call == "noalloc":
        row_ptr, col = _csr(*x)
        n = x[2]
        return {"call": call, "row_ptr": row_ptr, "col": col, "n": n,
                "tri": torch.empty(n, dtype=torch.uint64, device="cuda"),
                "numer": torch.empty(n, dtype=torch.uint64, device="cuda"),
                "tc": torch.empty(n, dtype=torch.float64, device="cuda")}
    reqs = [{"src": _pinned(s, torch.int32), "dst": _pinned(d, torch.int32), "n": n,
             "tri": torch.empty(n, dtype=torch.uint64, pin_memory=True),
             "tc": torch.empty(n, dtype=torch.float64, pin_memory=True)} for s, d, n in x]
    return {"call": call, "server": tc.Server(), "requests": reqs}


def _whole(t):
    """64-bit counts as the signed type that torch computes with (the same bytes)."""
    return t.view(torch.int64)


def run(state):
    call = state["call"]
    if call == "full":
        r = tc.triangle_centrality(state["src"], state["dst"], state["n"])
        return {"tri": _whole(r["tri"]), "flag": r["flag"], "total": r["total"], "numer": _whole(r["numer"]),
                "tc": r["tc"], "edge_u": r["edge_u"], "edge_v": r["edge_v"]}
    if call == "recount":
        tri, flag, total, _ = state["graph"].count()
        numer, cent, _, _ = state["graph"].centrality()
        return {"tri": _whole(tri), "flag": flag, "total": total, "numer": _whole(numer), "tc": cent}
    if call == "edges":
        tri, et, total, _ = state["graph"].edge_triangles()
        return {"tri": _whole(tri), "edge_tri": et.view(torch.int32), "total": total}
    if call in ("batch", "rerun"):
        b = state["batch"] if call == "rerun" else tc.Batch(*state["set"])
        o = b.run()
        if call == "batch":
            b.close()
        return {"tri": _whole(o["tri"]), "flag": o["flag"], "numer": _whole(o["numer"]), "tc": o["tc"],
                "totals": _whole(o["totals"])}
    if call == "noalloc":
        tc.tc_csr_centrality_noalloc(state["row_ptr"], state["col"], state["n"], tri=state["tri"],
                                     numer=state["numer"], tc=state["tc"])
        return {"tri": _whole(state["tri"]), "numer": _whole(state["numer"]), "tc": state["tc"]}
    srv = state["server"]
    ids = {srv.submit(q["src"], q["dst"], q["n"], q["tri"], q["tc"]): k for k, q in enumerate(state["requests"])}
    totals = [0] * len(ids)
    for info in srv.wait_all():
        totals[ids[info["id"]]] = info["triangles"]
    return {"tri": [_whole(q["tri"]) for q in state["requests"]], "tc": [q["tc"] for q in state["requests"]],
            "totals": np.array(totals, dtype=np.int64)}


# ------------------------------------------------------------- what it needs
def _rmat_edges(pairs):
    """Distinct undirected edges that `pairs` R-MAT pairs surely hold: their
    expected number less five standard deviations.  With b = c a vertex
    pair's probability depends only on how often each quadrant is taken."""
    a, b, _ = ABC
    d = 1.0 - a - 2 * b
    s, total = _scale(pairs), 0.0
    for i in range(s + 1):                 # levels in quadrant a
        for j in range(1, s + 1 - i):      # levels in quadrants b and c: 2^j ways, half of them u < v
            ways = math.comb(s, i) * math.comb(s - i, j) * 2.0 ** (j - 1)
            total += ways * -math.expm1(pairs * math.log1p(-2 * a**i * b**j * d ** (s - i - j)))
    return max(1, int(total - 5 * math.sqrt(total)))


def work(case):
    """Each input read once, each output written once (integer work: no flops)."""
    call = case["call"]
    if call in ("batch", "rerun"):
        # mean n of the log-uniform law; 5 edges a vertex in one half, about 1.3 in the other
        n = case["count"] * (case["n_max"] - 32) / math.log(case["n_max"] / 32)
        m = 3.1 * n
        return {"bytes": 24 * n + m + 8 * case["count"] + 8 * m, "flops": 0}
    if call == "serve":
        p = case["count"] * (case["pairs_max"] - 1000) / math.log(case["pairs_max"] / 1000)
        return {"bytes": 8 * p + 16 * p / 12, "flops": 0}
    if case["graph"] == "rmat":
        p, n, m = case["pairs"], 1 << _scale(case["pairs"]), _rmat_edges(case["pairs"])
    else:
        n, m = case["side"] ** 2, _grid_edges(case["side"])
        p = 1.05 * m
    if call == "full":      # pairs; △, numerator and TC; flags and edge list
        return {"bytes": 2 * p * case["ids"] / 8 + 24 * n + 9 * m, "flops": 0}
    if call == "recount":   # both ends of every edge once; △, numerator, TC and flags
        return {"bytes": 8 * m + 24 * n + m, "flops": 0}
    if call == "edges":
        return {"bytes": 8 * m + 8 * n + 4 * m, "flops": 0}
    return {"bytes": 8 * n + 8 * m + 24 * n, "flops": 0}   # noalloc


# --------------------------------------------------------------- in 64 bits
def _edge_counts(u, v, n):
    """Triangles on every edge (u < v, sorted): every pair of higher
    neighbours (degree order) of a vertex looked up among the edges."""
    m = len(u)
    deg = torch.bincount(torch.cat([u, v]), minlength=n)
    rank = torch.empty(n, dtype=torch.int64, device="cuda")
    rank[torch.sort(deg, stable=True).indices] = torch.arange(n, device="cuda")
    ru, rv = rank[u], rank[v]
    key, order = torch.sort(torch.minimum(ru, rv) * n + torch.maximum(ru, rv))
    lo, hi = key // n, key % n
    after = torch.bincount(lo, minlength=n).cumsum(0)[lo] - 1 - torch.arange(m, device="cuda")
    ends = after.cumsum(0)
    if m and int(ends[-1]) > MAX_EXACT_WEDGES:
        return None
    t = torch.zeros(m, dtype=torch.int64, device="cuda")
    one = torch.ones(1, dtype=torch.int64, device="cuda")
    at = 0
    while at < m:
        done = int(ends[at - 1]) if at else 0
        to = max(at + 1, int(torch.searchsorted(ends, done + (1 << 26), right=True)))
        g, j = _spread(after[at:to])
        i = at + g
        k = i + 1 + j
        q = hi[i] * n + hi[k]
        p = torch.searchsorted(key, q).clamp_(max=m - 1)
        hit = key[p] == q
        for x in (i, k, p):
            x = x[hit]
            t.index_add_(0, x, one.expand(x.shape))
        at = to
    out = torch.empty_like(t)
    out[order] = t
    return out


def _results(u, v, n, group=None):
    """(△ per vertex, triangles per edge, numerator, TC, sums) in whole
    numbers and one division; `group`: the graph of each vertex."""
    t = _edge_counts(u, v, n)
    if t is None:
        return None
    tri = torch.zeros(n, dtype=torch.int64, device="cuda").index_add_(0, u, t).index_add_(0, v, t) // 2
    w = torch.where(t > 0, 1, 3)
    numer = tri.clone().index_add_(0, u, w * tri[v]).index_add_(0, v, w * tri[u])
    if group is None:
        den = tri.sum()
        return tri, t, numer, numer.double() / den.double(), den
    den = torch.zeros(int(group[-1]) + 1, dtype=torch.int64, device="cuda").index_add_(0, group, tri)
    return tri, t, numer, numer.double() / den[group].double(), den


def exact(case, seed):
    x = _inputs(case, seed)
    if case["call"] == "serve":
        rs = [_results(*_distinct(*g), g[2]) for g in x]
        if any(r is None for r in rs):
            return None
        return {"tri": [r[0] for r in rs], "tc": [r[3] for r in rs],
                "totals": torch.stack([r[4] for r in rs]) // 3}
    if case["graph"] == "set":
        src, dst, off, nv = x
        voff = np.concatenate([[0], np.cumsum(nv)])
        shift = torch.repeat_interleave(torch.from_numpy(voff[:-1]).cuda(), torch.from_numpy(np.diff(off)).cuda())
        n = int(voff[-1])
        u, v = _distinct(src + shift, dst + shift, n)
        group = torch.repeat_interleave(torch.arange(len(nv), device="cuda"), torch.from_numpy(nv).cuda())
        r = _results(u, v, n, group)
        return r and {"tri": r[0], "flag": (r[1] > 0).to(torch.uint8), "numer": r[2], "tc": r[3], "totals": r[4] // 3}
    n = x[2]
    u, v = _distinct(*x)
    r = _results(u, v, n)
    if r is None:
        return None
    tri, t, numer, cent, den = r
    flag, total = (t > 0).to(torch.uint8), den // 3
    if case["call"] == "edges":
        return {"tri": tri, "edge_tri": t.to(torch.int32), "total": total}
    if case["call"] == "noalloc":
        return {"tri": tri, "numer": numer, "tc": cent}
    out = {"tri": tri, "flag": flag, "total": total, "numer": numer, "tc": cent}
    if case["call"] == "full":
        out.update(edge_u=u.to(torch.int32), edge_v=v.to(torch.int32))
    return out
