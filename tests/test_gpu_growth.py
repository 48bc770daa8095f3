"""Graphs of low degree whose searches have few steps of very many entries
(random and power-law graphs, a grid of three dimensions) do not take the
kernels over adjacency blocks where those are slower, and nearest-neighbour
graphs with long rows do not take the power-law graphs' team sizes."""

import numpy as np
import pytest

import oracle
from paper_2506_16488_gb300 import ppsp
from workloads import CSRGraph, clique_pairs, csr_from_undirected, grid_graph, random_pairs, rmat_graph, road_like_graph

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


def graph_of(n, u, v, seed):
    lo, hi = np.minimum(u, v), np.maximum(u, v)
    key = np.unique((lo.astype(np.int64) * n + hi)[lo != hi])
    w = np.random.default_rng(seed).integers(1, 1001, key.size).astype(np.uint32)
    off, tgt, wt = csr_from_undirected(n, key // n, key % n, w)
    return CSRGraph(n=n, offsets=off, targets=tgt, weights=wt, lcc=np.flatnonzero(np.diff(off) >= 2).astype(np.uint32))


def random_graph(n, deg, seed):
    rng = np.random.default_rng(seed)
    return graph_of(n, *rng.integers(0, n, (2, int(n * deg / 2))), seed)


def cube(side, seed):
    i = np.arange(side ** 3).reshape(side, side, side)
    u = np.r_[i[:-1].ravel(), i[:, :-1].ravel(), i[:, :, :-1].ravel()]
    v = np.r_[i[1:].ravel(), i[:, 1:].ravel(), i[:, :, 1:].ravel()]
    return graph_of(side ** 3, u, v, seed)


CASES = [  # graph, mode, queries, strategy, whether the kernels over adjacency blocks run
    ("random17", "et", 8, "plain_star", False), ("random17", "et", 1, "plain", False),
    ("random17", "bids", 8, "plain_star", True), ("random17", "bids", 400, "plain_star", False),
    ("random17", "et", 400, "plain_star", False), ("random17", "bids", 6, "clique", True),
    ("random15", "et", 8, "plain_star", False), ("random15", "et", 400, "plain_star", True),
    ("random15", "bids", 400, "plain_star", True), ("random12", "et", 8, "plain_star", True),
    ("cube40", "bids", 8, "plain_star", False), ("cube40", "bids", 400, "plain_star", True),
    ("cube40", "bids", 6, "clique", False),
    ("rmat13", "bids", 8, "plain_star", False), ("rmat13", "bids", 400, "plain_star", False),
    ("road200", "et", 8, "plain_star", True), ("grid64", "bids", 8, "plain_star", True),
]
GRAPHS = {"random17": lambda: random_graph(1 << 17, 4, 1), "random15": lambda: random_graph(1 << 15, 5, 2),
          "random12": lambda: random_graph(1 << 12, 4, 3), "cube40": lambda: cube(40, 4),
          "rmat13": lambda: rmat_graph(13, seed=5, edge_factor=3), "road200": lambda: road_like_graph(200, seed=6),
          "grid64": lambda: grid_graph(64, seed=7)}


@pytest.mark.parametrize("name", list(GRAPHS))
def test_kernel_by_growth(name):
    g = GRAPHS[name]()
    assert g.targets.size <= 6 * g.n
    with ppsp.Graph.from_csr(g, with_coords=False) as G:
        for _, mode, k, strategy, blocks in [c for c in CASES if c[0] == name]:
            if strategy == "clique":
                pairs, strategy = clique_pairs(g, k, 8), "multi"
            else:
                pairs = random_pairs(g, k, 9)
            with G.plan(pairs, mode=mode, strategy=strategy) as p:
                shape = p.launch_shape()
            assert (shape["kernel"] in ("bucket", "bucket_teams", "clusters")) == blocks, (mode, k, strategy, shape)
            want = oracle.pairs(g.offsets, g.targets, g.weights, pairs[:40])
            got = G.batch(pairs, mode=mode, strategy=strategy)
            assert np.array_equal(got[:40], want), (mode, k, strategy)


@pytest.mark.parametrize("side,seed", [(150, 21), (300, 22), (600, 23), (1000, 24)])
def test_road_graphs_in_device_order(side, seed):
    g = road_like_graph(side, seed=seed)
    for directed in (False, True):
        with ppsp.Graph.from_csr(g, undirected=not directed) as G:
            for mode, k in (("bidastar", 5), ("et", 200)):
                with G.plan(random_pairs(g, k, 25), mode=mode, strategy="plain_star") as p:
                    assert p.launch_shape()["kernel"] in ("bucket", "clusters"), (mode, k)


def test_nearest_neighbour_graph_keeps_small_teams():
    side, rng = 400, np.random.default_rng(10)
    i = np.arange(side * side).reshape(side, side)  # the eight neighbours of each cell
    u = np.r_[i[:, :-1].ravel(), i[:-1].ravel(), i[:-1, :-1].ravel(), i[:-1, 1:].ravel()]
    v = np.r_[i[:, 1:].ravel(), i[1:].ravel(), i[1:, 1:].ravel(), i[1:, :-1].ravel()]
    g = graph_of(side * side, u, v, 11)
    assert g.targets.size > 6 * g.n and g.targets.size > 1 << 20
    pairs = random_pairs(g, 24, 12)
    with ppsp.Graph.from_csr(g) as G:
        with G.plan(pairs, mode="bids", strategy="plain_star") as p:
            shape = p.launch_shape()
        assert (shape["kernel"], shape["block_threads"], shape["teams"]) == ("general", 512, 24), shape
        got = G.batch(pairs, mode="bids", strategy="plain_star")
        assert np.array_equal(got, oracle.pairs(g.offsets, g.targets, g.weights, pairs))
