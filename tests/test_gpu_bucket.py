"""The bucketed kernel over adjacency blocks, at the sizes where it can go
wrong: degrees around the block's four edges and a hub's hand-over to the whole
CTA, buckets that outgrow shared memory, the overflow region and the far list,
both directions of a directed graph, and distances at the width's limit."""

import numpy as np
import pytest

import oracle
from paper_2506_16488_gb300 import ppsp
from workloads import CSRGraph, csr_from_undirected, one_way_graph, random_pairs

pytestmark = pytest.mark.gpu

MODES = ("bids", "bidastar", "astar", "et")


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


def hub_graph(n, degrees, seed, extra=0):
    """A random tree-like graph with coordinates (average degree below four)
    and a vertex of about each of the given degrees; `extra` isolated vertices."""
    rng = np.random.default_rng(seed)
    v = np.arange(1, n)
    u = np.maximum(0, v - rng.integers(1, 60, n - 1))
    hubs = rng.choice(n, len(degrees), replace=False)
    for h, d in zip(hubs, degrees):
        u, v = np.r_[u, np.full(d, h)], np.r_[v, rng.choice(n, d, replace=False)]
    lo, hi = np.minimum(u, v), np.maximum(u, v)
    key = np.unique((lo * n + hi)[lo != hi])
    lo, hi = key // n, key % n
    xy = rng.uniform(0, 100, (n + extra, 2)).astype(np.float32)
    length = np.sqrt(((xy[lo].astype(np.float64) - xy[hi]) ** 2).sum(1))
    w = (np.rint(1000 * length).astype(np.int64) + rng.integers(1, 3000, lo.size)).astype(np.uint32)
    off, tgt, wt = csr_from_undirected(n + extra, lo, hi, w)
    pairs = np.concatenate([np.stack([np.repeat(hubs[:3], 4), rng.integers(0, n, 12)], 1), rng.integers(0, n, (30, 2))])
    return CSRGraph(n=n + extra, offsets=off, targets=tgt, weights=wt, coords=xy,
                    lcc=np.arange(n, dtype=np.uint32)), pairs.astype(np.uint32)


DEGREES = (3, 4, 5, 7, 8, 9, 12, 36, 37, 40, 41, 300, 1500)


@pytest.mark.parametrize("bits", [32, 64])
@pytest.mark.parametrize("delta", [0, 40, 1 << 40])
def test_degrees_around_the_block(bits, delta):
    g, pairs = hub_graph(4000, DEGREES, seed=31)
    want = oracle.pairs(g.offsets, g.targets, g.weights, pairs)
    with ppsp.Graph.from_csr(g) as G:
        for mode in MODES:
            for block in (256, 512, 1024):
                got = G.batch(pairs, mode=mode, strategy="plain_star", dist_bits=bits, delta=delta, block_threads=block)
                assert np.array_equal(got, want), (mode, block)
            assert np.array_equal(G.batch(pairs, mode=mode, strategy="vc", dist_bits=bits, delta=delta), want), mode
        for mode in MODES:
            for q in (0, 5, 20):
                st, d, path, _ = G.query_path(int(pairs[q, 0]), int(pairs[q, 1]), mode=mode, dist_bits=bits, delta=delta)
                assert st == ppsp.OK and d == int(want[q])
                if path is not None and len(path):
                    assert path[0] == pairs[q, 0] and path[-1] == pairs[q, 1]
                    assert oracle.path_weight(g.offsets, g.targets, g.weights, path) == d


@pytest.mark.parametrize("keep", [0.0, 0.6])
def test_directed_degrees(keep):
    g, pairs = hub_graph(3000, DEGREES, seed=32, extra=5)
    d = one_way_graph(g, keep, seed=33)
    pairs = np.r_[pairs, [[1, 3001], [3002, 7]]].astype(np.uint32)  # unreachable
    want = oracle.pairs(d.offsets, d.targets, d.weights, pairs)
    with ppsp.Graph.from_csr(d, undirected=False) as G:
        for mode in MODES:
            assert np.array_equal(G.batch(pairs, mode=mode, strategy="plain_star"), want), mode
            assert np.array_equal(G.batch(pairs, mode=mode, strategy="vc", dist_bits=64), want), mode


@pytest.mark.parametrize("delta,ring", [(1 << 40, 1), (1 << 40, 0), (1, 1), (60, 3)])
def test_overflow_far_list_and_spills(delta, ring):
    # a hub of 30,000 edges: one relaxation fills a bucket past shared memory
    # and its overflow region (large increment) or the far list (small one)
    g, pairs = hub_graph(40000, (30000, 9000, 200), seed=34)
    pairs = pairs[::3]
    want = oracle.pairs(g.offsets, g.targets, g.weights, pairs)
    with ppsp.Graph.from_csr(g) as G:
        for mode in MODES if delta != 1 else ("bids",):
            for bits in (32, 64):
                got = G.batch(pairs, mode=mode, strategy="plain_star", delta=delta, ring_entries=ring, dist_bits=bits)
                assert np.array_equal(got, want), (mode, bits)


def test_disconnected_pairs_and_width_limit():
    # two paths of heavy edges: unreachable pairs, and sums at the 32-bit limit
    w = 1 << 28
    n = 40
    u = np.r_[np.arange(0, 19), np.arange(20, 39)]
    off, tgt, wt = csr_from_undirected(n, u, u + 1, np.full(u.size, w, dtype=np.uint32))
    pairs = np.array([[0, 10], [0, 15], [3, 25], [39, 30], [20, 0], [5, 5]], dtype=np.uint32)
    want = oracle.pairs(off, tgt, wt, pairs)
    with ppsp.Graph(off, tgt, wt) as G:
        for mode in ("bids", "et"):
            assert np.array_equal(G.batch(pairs, mode=mode, strategy="plain_star", dist_bits=64), want), mode
        # 16 edges of 2^28 do not fit 32 bits: an error, not a wrong answer
        st, _ = G.batch_status(np.array([[0, 17]], dtype=np.uint32), mode="et", strategy="plain_star")
        assert st == ppsp.ERR_OVERFLOW
        got = G.batch(np.array([[0, 7], [22, 29]], dtype=np.uint32), mode="bids", strategy="plain_star")
        assert got.tolist() == [7 * w, 7 * w]


@pytest.mark.parametrize("bits", [32, 64])
@pytest.mark.parametrize("shape", ["clique3", "clique9", "star64", "mixed"])
def test_groups_of_several_searches(shape, bits):
    g, pairs = hub_graph(3000, DEGREES, seed=35, extra=4)
    rng = np.random.default_rng(36)

    def clique(k):
        v = rng.choice(3000, k, replace=False)
        i, j = np.triu_indices(k, 1)
        return np.stack([v[i], v[j]], 1)

    v = rng.choice(3000, 65, replace=False)
    star = np.stack([np.full(63, v[0]), v[1:64]], 1)
    p = {"clique3": clique(3), "clique9": clique(9), "star64": star,
         "mixed": np.concatenate([pairs, clique(5), clique(3), star, [[3001, 1], [1, 17], [17, 3002]]])}[shape]
    p = p.astype(np.uint32)
    d = one_way_graph(g, 0.3, seed=37)
    for graph, directed in ((g, False), (d, True)):
        want = oracle.pairs(graph.offsets, graph.targets, graph.weights, p)
        with ppsp.Graph.from_csr(graph, undirected=not directed) as G:
            for mode in ("bids", "bidastar"):
                for kw in ({}, {"delta": 30}, {"delta": 1 << 40, "ring_entries": 1}, {"block_threads": 512},
                           {"block_threads": 256, "max_ctas": 66}, {"max_ctas": 2}):
                    for _ in range(2):  # the second batch finds the slots as the first left them
                        got = G.batch(p, mode=mode, strategy="multi", dist_bits=bits, **kw)
                        assert np.array_equal(got, want), (directed, mode, kw)


@pytest.mark.parametrize("bits", [32, 64])
@pytest.mark.parametrize("k", [1, 2, 5, 30])
def test_clusters(k, bits):
    """Few queries of large steps run on clusters of CTAs (2, 4 or 8 by the
    number of queries): the same answers, hubs, overflow and far lists included."""
    g, pairs = hub_graph(60000, DEGREES + (20000,), seed=38, extra=3)
    pairs = np.r_[pairs[:k - 1], pairs[-1:]] if k > 1 else pairs[:1]
    lost = np.array([[5, 60001]], dtype=np.uint32)
    star = np.stack([np.full(12, pairs[0, 0]), np.arange(100, 112)], 1).astype(np.uint32)
    d = one_way_graph(g, 0.2, seed=39)
    for graph, directed in ((g, False), (d, True)):
        want, far, st = (oracle.pairs(graph.offsets, graph.targets, graph.weights, p) for p in (pairs, lost, star))
        for coords in (True, False):
            with ppsp.Graph.from_csr(graph, undirected=not directed, with_coords=coords) as G:
                for mode in MODES if coords else ("bids", "et"):
                    for kw in ({}, {"delta": 1 << 40}, {"ring_entries": 1}, {"delta": 200, "ring_entries": 2},
                               {"max_ctas": 3}):
                        for _ in range(2):
                            got = G.batch(pairs, mode=mode, strategy="plain_star", dist_bits=bits, **kw)
                            assert np.array_equal(got, want), (directed, mode, kw)
                    assert G.query(*pairs[0].tolist(), mode=mode, dist_bits=bits) == int(want[0])
                    assert np.array_equal(G.batch(lost, mode=mode, strategy="plain_star", dist_bits=bits), far)
                    assert np.array_equal(G.batch(star, mode=mode, strategy="vc", dist_bits=bits), st)
