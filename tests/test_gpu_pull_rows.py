"""Pull-then-push relaxation on graphs whose rows are sorted by weight and cut
at the prune bound: the pull lowers a vertex's distance after its row was read,
so edges that were too long for the old distance have to be pushed too."""

import numpy as np
import pytest

import oracle
from paper_2506_16488_gb300 import ppsp
from workloads import CSRGraph, clique_pairs, csr_from_undirected, random_pairs, rmat_graph, star_pairs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


def detour_graph():
    """s-u 10, s-x 1, x-u 1, u-t 6, s-t 15, and a clique elsewhere that makes
    the average degree long-row: u is extracted at 10 with mu = 15, pulls 2
    from x, and only then reaches t at 8."""
    s, u, x, t, n = 0, 1, 2, 3, 24
    iu, ju = np.triu_indices(20, 1)
    a = np.r_[[s, s, x, u, s], iu + 4]
    b = np.r_[[u, x, u, t, t], ju + 4]
    w = np.r_[[10, 1, 1, 6, 15], np.full(iu.size, 50)].astype(np.uint32)
    off, tgt, wt = csr_from_undirected(n, a, b, w)
    return CSRGraph(n=n, offsets=off, targets=tgt, weights=wt, lcc=np.arange(n, dtype=np.uint32))


@pytest.mark.parametrize("mode", ["et", "bids"])
@pytest.mark.parametrize("delta", [0, 1, 10 ** 7])
def test_detour_found_by_the_pull(mode, delta):
    g = detour_graph()
    with ppsp.Graph.from_csr(g) as G:
        for team in (2, 8):
            for pull in (False, True):
                assert G.query(0, 3, mode=mode, pull_push=pull, team_ctas=team, delta=delta) == 8, (team, pull)
                got = G.batch([[0, 3], [1, 0]], mode=mode, strategy="vc", pull_push=pull, team_ctas=team, delta=delta)
                assert got.tolist() == [8, 2], (team, pull)


@pytest.mark.parametrize("bits", [32, 64])
@pytest.mark.parametrize("wmax", [30, 65535])
def test_pull_on_long_rows(bits, wmax):
    g = rmat_graph(12, seed=51)
    lo = np.minimum(np.repeat(np.arange(g.n), np.diff(g.offsets.astype(np.int64))), g.targets)
    hi = np.maximum(np.repeat(np.arange(g.n), np.diff(g.offsets.astype(np.int64))), g.targets)
    w = ((lo * 7919 + hi * 104729) % wmax + 1).astype(np.uint32)  # the same both ways
    g = CSRGraph(n=g.n, offsets=g.offsets, targets=g.targets, weights=w, lcc=g.lcc)
    pairs = np.concatenate([random_pairs(g, 24, 52), clique_pairs(g, 6, 53), star_pairs(g, 9, 54)])
    want = oracle.pairs(g.offsets, g.targets, g.weights, pairs)
    with ppsp.Graph.from_csr(g) as G:
        for mode in ("bids", "et"):
            for strategy in ("multi", "plain_star", "vc"):
                for delta in (0, wmax, 10 ** 7):
                    for frontier in ("auto", "sparse", "dense"):
                        got = G.batch(pairs, mode=mode, strategy=strategy, pull_push=True, team_ctas=2, big_team_ctas=2,
                                      delta=delta, frontier=frontier, dist_bits=bits)
                        assert np.array_equal(got, want), (mode, strategy, delta, frontier)
