"""The kernels over adjacency blocks, one CTA, clusters of two, four and eight
and one CTA per search, on a road-like graph with hubs: which of them a plan
takes is asserted (Plan.launch_shape), so that none goes untested."""

import numpy as np
import pytest
import torch

import oracle
from paper_2506_16488_gb300 import ppsp
from workloads import CSRGraph, csr_from_undirected, one_way_graph

pytestmark = pytest.mark.gpu

MODES = ("bids", "bidastar", "astar", "et")
DEGREES = (5, 7, 8, 9, 12, 36, 37, 40, 41, 300, 1500, 15000)


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


def grid_with_hubs(side, degrees, seed, extra=0):
    """A jittered grid with a tenth of its edges deleted; each hub is joined to
    vertices of a square around it by edges of nearly the same weight (a step
    that takes a hub inserts thousands of entries into a few buckets).  `extra`
    isolated vertices at the end."""
    rng = np.random.default_rng(seed)
    n = side * side
    ids = np.arange(n).reshape(side, side)
    u = np.r_[ids[:, :-1].ravel(), ids[:-1].ravel()]
    v = np.r_[ids[:, 1:].ravel(), ids[1:].ravel()]
    keep = rng.random(u.size) >= 0.1
    u, v = u[keep], v[keep]
    xy = (np.stack([np.arange(n + extra) % side, np.arange(n + extra) // side], 1)
          + rng.uniform(-0.3, 0.3, (n + extra, 2))).astype(np.float32)
    hubs = rng.choice(n, len(degrees), replace=False)
    flat = np.zeros(u.size, dtype=np.int64)
    for h, d in zip(hubs, degrees):
        half = min(side // 2, int(np.sqrt(d) / 2) + 4)
        x0, y0 = min(max(h % side - half, 0), side - 2 * half), min(max(h // side - half, 0), side - 2 * half)
        near = ids[y0:y0 + 2 * half, x0:x0 + 2 * half].ravel()
        near = rng.choice(near, min(d, near.size), replace=False)
        u, v = np.r_[u, np.full(near.size, h)], np.r_[v, near]
        flat = np.r_[flat, rng.integers(700 * half, 700 * half + 300, near.size)]
    lo, hi = np.minimum(u, v), np.maximum(u, v)
    key, first = np.unique(lo * n + hi, return_index=True)
    lo, hi, flat = key // n, key % n, flat[first]
    ok = lo != hi
    lo, hi, flat = lo[ok], hi[ok], flat[ok]
    length = np.sqrt(((xy[lo].astype(np.float64) - xy[hi]) ** 2).sum(1))
    w = np.where(flat > 0, flat, np.rint(1000 * length) + 1).astype(np.uint32)
    off, tgt, wt = csr_from_undirected(n + extra, lo, hi, w)
    g = CSRGraph(n=n + extra, offsets=off, targets=tgt, weights=wt, coords=xy, lcc=np.arange(n, dtype=np.uint32))
    return g, hubs


def check(G, pairs, want, expect=None, **kw):
    """Both runs of a plan (the second finds the slots as the first left them)
    against the oracle; its kernel."""
    out = torch.zeros(len(pairs), dtype=torch.int64, device="cuda")
    with G.plan(pairs, **kw) as p:
        shape = p.launch_shape()
        if expect:
            assert (shape["kernel"], shape["cluster"]) == expect, (shape, kw)
        for _ in range(2):
            out.fill_(7)
            torch.cuda.synchronize()
            p.run(out.data_ptr())
            p.sync()
            assert np.array_equal(out.cpu().numpy().view(np.uint64), want), (shape, kw)
    return shape


@pytest.fixture(scope="module")
def hubs700():
    g, hubs = grid_with_hubs(700, DEGREES, seed=81, extra=3)
    rng = np.random.default_rng(82)
    pairs = np.concatenate([np.stack([hubs[-6:], rng.integers(0, 490000, 6)], 1), rng.integers(0, 490000, (66, 2))])
    pairs = pairs[rng.permutation(len(pairs))].astype(np.uint32)
    pairs[0, 0] = hubs[-1]
    d = one_way_graph(g, 0.2, seed=83)
    return [(x, not und, pairs, oracle.pairs(x.offsets, x.targets, x.weights, pairs)) for x, und in ((g, True), (d, False))]


@pytest.mark.parametrize("bits", [32, 64])
@pytest.mark.parametrize("coords", [False, True])
@pytest.mark.parametrize("directed", [False, True])
def test_cluster_sizes(hubs700, directed, coords, bits):
    g, _, pairs, want = hubs700[int(directed)]
    mean = int(g.weights.mean())
    seen = set()
    with ppsp.Graph.from_csr(g, undirected=not directed, with_coords=coords) as G:
        for mode in MODES if coords else ("bids", "et"):
            for k in (1, 6, 30, 60):
                for kw in ({}, {"delta": 2 * mean}, {"ring_entries": 1}, {"delta": 200, "ring_entries": 2}, {"max_ctas": 3}):
                    if kw.get("delta") == 200 and k > 6:
                        continue
                    s = check(G, pairs[:k], want[:k], mode=mode, strategy="plain_star", dist_bits=bits, **kw)
                    if s["kernel"] == "clusters":
                        seen.add(s["cluster"])
                        assert s["cluster"] <= (2 if "max_ctas" in kw else 8)
            assert G.query(*pairs[0].tolist(), mode=mode, dist_bits=bits) == int(want[0])
            # unreachable (the disconnected exit), and one search with many targets
            lost = np.array([[5, 490001], [490002, 9]], dtype=np.uint32)
            check(G, lost, np.full(2, ppsp.INF, dtype=np.uint64), mode=mode, strategy="plain_star", dist_bits=bits)
            star = np.stack([np.full(12, pairs[0, 0]), pairs[:12, 1]], 1).astype(np.uint32)
            st = oracle.pairs(g.offsets, g.targets, g.weights, star)
            check(G, star, st, mode=mode, strategy="vc", dist_bits=bits)
    if not coords:
        assert seen == {2, 4, 8}, seen


@pytest.mark.parametrize("bits", [32, 64])
@pytest.mark.parametrize("directed", [False, True])
def test_one_cta_and_one_cta_per_search(hubs700, directed, bits):
    g, _, pairs, want = hubs700[int(directed)]
    rng = np.random.default_rng(84)
    x, y = rng.integers(0, 690, (2, 170))
    near = np.stack([y * 700 + x, (y + rng.integers(0, 9, 170)) * 700 + x + rng.integers(1, 9, 170)], 1).astype(np.uint32)
    near_want = oracle.pairs(g.offsets, g.targets, g.weights, near)
    many, many_want = np.concatenate([near, pairs]), np.concatenate([near_want, want])
    v = rng.choice(490000, 9, replace=False)
    i, j = np.triu_indices(9, 1)
    clique = np.stack([v[i], v[j]], 1).astype(np.uint32)
    cw = oracle.pairs(g.offsets, g.targets, g.weights, clique)
    with ppsp.Graph.from_csr(g, undirected=not directed) as G:
        for mode in MODES:
            for kw in ({"max_ctas": 150}, {"block_threads": 256, "max_ctas": 200}, {"ring_entries": 1, "max_ctas": 100}):
                check(G, many, many_want, ("bucket", 1), mode=mode, strategy="plain_star", dist_bits=bits, **kw)
            for kw in ({"delta": 1 << 40, "ring_entries": 1}, {"delta": 300, "ring_entries": 3}):
                check(G, near, near_want, ("bucket", 1), mode=mode, strategy="plain_star", dist_bits=bits, max_ctas=40, **kw)
        for mode in ("bids", "bidastar"):
            for kw in ({}, {"ring_entries": 1}, {"delta": 300}):
                check(G, clique, cw, ("bucket_teams", 1), mode=mode, strategy="multi", dist_bits=bits, **kw)
