"""The queue / bitmap path on graphs with long rows: rows sorted by weight and
cut at the prune bound, rows shared by a team in pieces, tiles smaller than a
CTA."""

import numpy as np
import pytest

import oracle
from paper_2506_16488_gb300 import ppsp
from workloads import clique_pairs, csr_from_undirected, one_way_graph, random_pairs, rmat_graph, star_pairs, CSRGraph

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


def hubs(n, degrees, seed, wmax):
    """Average degree above six, and rows around the piece size (2,048)."""
    rng = np.random.default_rng(seed)
    u, v = rng.integers(0, n, 4 * n), rng.integers(0, n, 4 * n)
    for h, d in enumerate(degrees):
        u, v = np.r_[u, np.full(d, h)], np.r_[v, rng.choice(n, d, replace=False)]
    lo, hi = np.minimum(u, v), np.maximum(u, v)
    key = np.unique((lo * n + hi)[lo != hi])
    w = rng.integers(1, wmax + 1, key.size).astype(np.uint32)
    off, tgt, wt = csr_from_undirected(n, key // n, key % n, w)
    return CSRGraph(n=n, offsets=off, targets=tgt, weights=wt, lcc=np.arange(n, dtype=np.uint32))


@pytest.mark.parametrize("wmax", [1, 9, 65535])
@pytest.mark.parametrize("bits", [32, 64])
def test_long_rows(bits, wmax):
    g = hubs(12000, (2030, 2040, 2050, 4090, 6150, 11900), seed=41, wmax=wmax)
    pairs = np.concatenate([random_pairs(g, 20, 42), [[0, 9], [1, 5], [5, 11000], [7, 7]], clique_pairs(g, 4, 43),
                            star_pairs(g, 9, 44)]).astype(np.uint32)
    want = oracle.pairs(g.offsets, g.targets, g.weights, pairs)
    with ppsp.Graph.from_csr(g) as G:
        for mode in ("bids", "et"):
            for strategy in ("auto", "multi", "vc", "plain"):
                for kw in ({}, {"team_ctas": 2, "block_threads": 256}, {"frontier": "sparse"}, {"frontier": "dense"},
                           {"delta": 1}, {"delta": 1 << 33, "team_ctas": 1}):
                    if kw.get("delta") == 1 and wmax > 9:
                        continue
                    got = G.batch(pairs, mode=mode, strategy=strategy, dist_bits=bits, **kw)
                    assert np.array_equal(got, want), (mode, strategy, kw)
            for q in (0, 3, 21):
                st, d, path, _ = G.query_path(int(pairs[q, 0]), int(pairs[q, 1]), mode=mode, dist_bits=bits)
                assert st == ppsp.OK and d == int(want[q])
                if path is not None and len(path):
                    assert oracle.path_weight(g.offsets, g.targets, g.weights, path) == d


def test_long_rows_directed():
    g = one_way_graph(rmat_graph(13, seed=45), 0.5, seed=46)
    pairs = np.concatenate([random_pairs(g, 30, 47), star_pairs(g, 8, 48)]).astype(np.uint32)
    want = oracle.pairs(g.offsets, g.targets, g.weights, pairs)
    with ppsp.Graph.from_csr(g, undirected=False) as G:
        for mode in ("bids", "et"):
            for strategy in ("auto", "multi", "vc", "plain_star"):
                assert np.array_equal(G.batch(pairs, mode=mode, strategy=strategy), want), (mode, strategy)


def test_overflow_is_still_reported_behind_the_cut():
    # rows sorted by weight: the cut must not hide a distance that does not fit
    n = 30
    iu, ju = np.triu_indices(n, 1)
    w = np.full(iu.size, 3_000_000_000, dtype=np.uint32)
    w[iu == 0] = 1
    off, tgt, wt = csr_from_undirected(n, iu, ju, w)
    with ppsp.Graph(off, tgt, wt) as G:
        pairs = np.array([[3, 7], [4, 9]], dtype=np.uint32)
        assert np.array_equal(G.batch(pairs, mode="et", dist_bits=64), [2, 2])
        assert G.batch(np.array([[0, 7]], dtype=np.uint32), mode="et", delta=1).tolist() == [1]
