"""Kernels at the sizes where their tiles, units and rules end: each case
against the oracle, bit for bit."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import graphgen as gg
import oracle
import paper_2105_00110_gb300 as tcg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    tcg.build()
    torch.cuda.init()


def csr_rows(rows):
    row_ptr = np.zeros(len(rows) + 1, np.int64)
    np.cumsum([len(r) for r in rows], out=row_ptr[1:])
    return row_ptr, np.array([c for r in rows for c in r], np.int32)


def noalloc(row_ptr, col, n):
    out = [torch.full((n,), 7, dtype=torch.int64, device="cuda").view(torch.uint64) for _ in range(2)]
    tc = torch.full((n,), 7.0, dtype=torch.float64, device="cuda")
    tcg.tc_csr_centrality_noalloc(torch.from_numpy(row_ptr).cuda(), torch.from_numpy(col).cuda(), n, *out, tc)
    return [x.cpu().numpy() for x in (*out, tc)]


def star(leaves):
    """A hub, its leaves and one triangle on it."""
    a = np.concatenate([np.zeros(leaves, np.int32), [1]]).astype(np.int32)
    b = np.concatenate([np.arange(1, leaves + 1), [2]]).astype(np.int32)
    return a, b, leaves + 1


@pytest.mark.parametrize("graph", [
    (np.zeros(0, np.int32), np.zeros(0, np.int32), 1),
    (np.array([0], np.int32), np.array([1], np.int32), 2),
    gg.complete_graph(17), gg.complete_graph(33),
    star(255), star(256), star(1000),            # rows around the gather's whole-CTA rows
    gg.gnp(65, 0.2, 5), gg.gnp(130, 0.5, 6),     # more than one bitmap word a row, ragged units
    gg.rmat(13, 16, seed=7), gg.rmat(15, 14, seed=8),   # units of 16 and of 32 entries
], ids=lambda g: "n%d-p%d" % (g[2], len(g[0])))
def test_allocation_free_units(graph):
    s, d, n = graph
    ref = oracle.run(s, d, n)
    tri, numer, tc = noalloc(ref["ptr"].astype(np.int64), ref["adj"].astype(np.int32), n)
    assert np.array_equal(tri, ref["tri"]) and np.array_equal(numer, ref["numer"])
    assert np.array_equal(tc, ref["tc"], equal_nan=True)


@pytest.mark.parametrize("rows", [
    [[0, 1], [0], []],                           # a loop
    [[1, 1], [0, 0]],                            # repeated entries
    [[1], [0], [3], []],                         # one-sided
    [[1, 2, 3, 4, 5], [0], [0], [], [], []],     # three of five one-sided
], ids=["loop", "repeat", "one-sided", "hub-one-sided"])
def test_allocation_free_rejects(rows):
    row_ptr, col = csr_rows(rows)
    if len(col) & 1:
        col, row_ptr = np.append(col, 0).astype(np.int32), np.append(row_ptr[:-1], len(col) + 1)
    tri, numer, tc = noalloc(row_ptr, col, len(rows))
    assert (tri.view(np.int64) == -1).all() and (numer.view(np.int64) == -1).all() and np.isnan(tc).all()


def check_full(src, dst, n):
    """One full pass against the oracle, and the plan's wedge count against
    the out-degrees of the degree order."""
    res = tcg.triangle_centrality(torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda(), n)
    ref = oracle.run(src, dst, n)
    assert res["total"] == ref["total"]
    for k in ("tri", "numer"):
        assert np.array_equal(res[k].cpu().numpy(), ref[k][:n]), k
    assert np.array_equal(res["tc"].cpu().numpy(), ref["tc"][:n], equal_nan=True)
    rows = np.repeat(np.arange(n, dtype=np.int64), np.diff(ref["ptr"]))
    keep = ref["adj"] > rows
    u, v = rows[keep], ref["adj"][keep].astype(np.int64)
    assert np.array_equal(res["edge_u"].cpu().numpy(), u) and np.array_equal(res["edge_v"].cpu().numpy(), v)
    assert np.array_equal(res["flag"].cpu().numpy(), ref["flag"][keep])
    deg = np.bincount(np.concatenate([u, v]), minlength=n)
    rank = np.empty(n, np.int64)
    rank[np.argsort(deg, kind="stable")] = np.arange(n)
    dh = np.bincount(np.minimum(rank[u], rank[v]), minlength=n)
    st = res["stats"]
    assert st["wedges"] == float((dh * (dh - 1) // 2).sum()) and st["max_out_degree"] == dh.max(initial=0)
    assert st["max_degree"] == deg.max(initial=0) and st["sum_out_degree_sq"] == float((dh * dh).sum())
    assert sum(st["class_wedges"]) == st["wedges"]
    return res


def wheels(*rims):
    """Hubs, each joined to every vertex of a cycle of its own; the hubs are
    chained."""
    src, dst, n = [], [], len(rims)
    for h, r in enumerate(rims):
        rim = np.arange(n, n + r)
        src += [np.full(r, h), rim]
        dst += [rim, np.roll(rim, 1)]
        n += r
    src.append(np.arange(1, len(rims)))
    dst.append(np.arange(len(rims) - 1))
    return np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32), n


# hub rows (degree above 4096) are walked in segments of 2048 positions
@pytest.mark.parametrize("rims", [(4093,), (4097,), (4098, 6144), (20001, 4100, 33), (8192, 8191, 8190)],
                         ids=lambda r: "-".join(map(str, r)))
def test_hub_rows(rims):
    check_full(*wheels(*rims))


def sort_inputs(kind, p):
    rng = np.random.default_rng(p)
    if kind == "uniform":                 # buckets of like size
        n = 1 << 21
        return rng.integers(0, n, p), rng.integers(0, n, p), n
    if kind == "one-pair":                # one key, p times: bits run out
        return np.full(p, 7), np.full(p, 3), 1 << 20
    if kind == "few-keys":                # a small key space, every key many times
        return rng.integers(0, 40, p), rng.integers(0, 40, p), 40
    if kind == "loops":                   # nothing left
        a = rng.integers(0, 1000, p)
        return a, a, 1000
    if kind == "star":                    # one row holds everything, in order
        return np.zeros(p, np.int64), np.arange(1, p + 1), p + 1
    if kind == "hubs":                    # rows of several sizes beside light ones
        n = 1 << 20
        hub = rng.choice([5, 6, 70000, 70001, n - 2], p)
        return np.where(rng.random(p) < 0.6, hub, rng.integers(0, n, p)), rng.integers(0, n, p), n
    if kind == "clustered":               # higher ends crowd together: crowded sub-bins
        n = 1 << 22
        a = rng.integers(0, 64, p)
        return a, 1000 + (np.abs(rng.normal(0, 40, p))).astype(np.int64), n
    n = 3_000_001                         # ragged: n above a power of two, wide keys
    return (rng.random(p) ** 3 * n).astype(np.int64), rng.integers(0, n, p), n


@pytest.mark.parametrize("ids", [np.int32, np.int64])
@pytest.mark.parametrize("kind,p", [("uniform", 1 << 19), ("uniform", (1 << 20) + 1), ("one-pair", 600_000),
                                    ("few-keys", 700_001), ("loops", 1 << 19), ("star", (1 << 20) - 1),
                                    ("hubs", 3_000_000), ("clustered", 1 << 20), ("ragged", 2_500_003),
                                    ("uniform", (1 << 19) - 1)])
def test_sorted_edges(kind, p, ids):
    src, dst, n = sort_inputs(kind, p)
    g = tcg.Graph(torch.from_numpy(src.astype(ids)).cuda(), torch.from_numpy(dst.astype(ids)).cuda(), n)
    lo, hi = np.minimum(src, dst).astype(np.int64), np.maximum(src, dst).astype(np.int64)
    key = np.unique((lo * n + hi)[lo != hi])
    u, v = (x.cpu().numpy() for x in g.edges())
    assert g.m == len(key) and np.array_equal(u, key // n) and np.array_equal(v, key % n)
    g.close()


def test_sort_rejects_a_bad_id():
    src = np.arange(1 << 19, dtype=np.int32) % 1000
    for at, bad in ((12345, 1000), ((1 << 19) - 1, -1)):
        dst = np.roll(src, 1)
        dst[at] = bad
        with pytest.raises(tcg.TCError) as e:
            tcg.Graph(torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda(), 1000)
        assert e.value.status == tcg.TC_ERR_INVALID_ARG


@pytest.mark.parametrize("scale,short", [(14, 1), (14, 0), (17, 0)])
def test_small_graph_rules(scale, short):
    # below 1024 vertices an SM a warp takes 4 rows of short runs instead of
    # 32; below 4096 wedges a warp's share warp items are split beyond the
    # target in the plan parameters, which holds once a caller sets it
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    s, d, n = gg.rmat(scale, seed=9)
    n = max(n, 1024 * sms - short)
    ref = oracle.run(s, d, n)
    g = tcg.Graph(torch.from_numpy(s).cuda(), torch.from_numpy(d).cuda(), n)
    try:
        st = g.stats()
        tri, flags, total, _ = g.count()
        numer, tc, _, _ = g.centrality()
        assert np.array_equal(tri.cpu().numpy(), ref["tri"]) and total == ref["total"]
        assert np.array_equal(numer.cpu().numpy(), ref["numer"])
        assert np.array_equal(tc.cpu().numpy(), ref["tc"], equal_nan=True)
        tcg.tc_set_plan_params(g.h, **tcg.tc_get_plan_params(g.h))
        again, _, _, _ = g.count()
        assert np.array_equal(again.cpu().numpy(), ref["tri"])
        assert (g.stats()["items"][2] < st["items"][2]) == (st["wedges"] / (64.0 * sms) < 4096.0)
    finally:
        g.close()
