"""Rows sorted by weight and cut at the prune bound: a candidate that does not
fit the distance width is still reported, and searches with a potential stay
exact."""

import numpy as np
import pytest

import oracle
from paper_2506_16488_gb300 import ppsp
from workloads import CSRGraph, clique_pairs, csr_from_undirected, random_pairs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("leaves", [30, 5000])  # u's row in one tile, and in pieces of 2,048
@pytest.mark.parametrize("kw", [{}, {"team_ctas": 1}, {"team_ctas": 2}, {"frontier": "dense"}])
def test_overflow_in_the_cut_part_of_a_row(leaves, kw):
    # s-t 2^31 sets mu before u (at 10) is taken; u's last edge ends above 2^32
    s, t, u, x = 0, 1, 2, 3
    n, rng = 4 + leaves, np.random.default_rng(55)
    a = np.r_[[s, s, u], np.full(leaves, u), rng.integers(4, n, 6 * leaves)]
    b = np.r_[[t, u, x], np.arange(4, n), rng.integers(4, n, 6 * leaves)]
    w = np.r_[[1 << 31, 10, (1 << 32) - 5], rng.integers(1, 100, leaves), np.full(6 * leaves, 1 << 30)]
    lo, hi = np.minimum(a, b), np.maximum(a, b)
    key, first = np.unique(lo * n + hi, return_index=True)
    ok = key // n != key % n
    off, tgt, wt = csr_from_undirected(n, (key // n)[ok], (key % n)[ok], w[first][ok].astype(np.uint32))
    assert tgt.size > 6 * n
    pairs = np.array([[s, t]], dtype=np.uint32)
    with ppsp.Graph(off, tgt, wt) as G:
        st, _ = G.batch_status(pairs, mode="et", dist_bits=32, strategy="plain_star", **kw)
        assert st == ppsp.ERR_OVERFLOW
        got = G.batch(pairs, mode="et", dist_bits=64, strategy="plain_star", **kw)
        assert np.array_equal(got, oracle.pairs(off, tgt, wt, pairs))


@pytest.mark.parametrize("bits", [32, 64])
@pytest.mark.parametrize("long_row", [0, 4500])
def test_potentials_on_long_rows(bits, long_row):
    side, rng = 90, np.random.default_rng(56)
    n = side * side
    i = np.arange(n).reshape(side, side)  # eight neighbours, and a hub
    u = np.r_[i[:, :-1].ravel(), i[:-1].ravel(), i[:-1, :-1].ravel(), i[:-1, 1:].ravel(), np.full(long_row, 4000)]
    v = np.r_[i[:, 1:].ravel(), i[1:].ravel(), i[1:, 1:].ravel(), i[1:, :-1].ravel(), rng.choice(n, long_row, replace=False)]
    lo, hi = np.minimum(u, v), np.maximum(u, v)
    key = np.unique((lo * n + hi)[lo != hi])
    lo, hi = key // n, key % n
    xy = (np.stack([np.arange(n) % side, np.arange(n) // side], 1) + rng.uniform(-0.3, 0.3, (n, 2))).astype(np.float32)
    length = np.sqrt(((xy[lo].astype(float) - xy[hi]) ** 2).sum(1))
    w = (np.ceil(1000 * length) + rng.integers(0, 4000, lo.size)).astype(np.uint32)
    off, tgt, wt = csr_from_undirected(n, lo, hi, w)
    assert tgt.size > 6 * n
    g = CSRGraph(n=n, offsets=off, targets=tgt, weights=wt, coords=xy, lcc=np.arange(n, dtype=np.uint32))
    pairs = np.concatenate([random_pairs(g, 40, 57), clique_pairs(g, 5, 58), [[4000, 17], [33, 4000]]]).astype(np.uint32)
    want = oracle.pairs(off, tgt, wt, pairs)
    with ppsp.Graph.from_csr(g) as G:
        for mode in ("astar", "bidastar"):
            for kw in ({}, {"team_ctas": 1}, {"team_ctas": 4}, {"frontier": "sparse"}, {"frontier": "dense", "delta": 400},
                       {"memo_potential": True, "team_ctas": 2}, {"strategy": "plain"}):
                got = G.batch(pairs, mode=mode, dist_bits=bits, **{"strategy": "plain_star", **kw})
                assert np.array_equal(got, want), (mode, kw)
        for mp in (False, True):
            got = G.batch(pairs, mode="bidastar", strategy="multi", multi_potential=mp, dist_bits=bits)
            assert np.array_equal(got, want), mp
