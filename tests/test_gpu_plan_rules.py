"""Rules of a plan's launch: CTA size and clusters where groups run one at a
time, on few CTAs or on explicit sizes, team_ctas = 1, little device memory,
and increments and estimates without a usable potential."""

import numpy as np
import pytest
import torch

import oracle
from paper_2506_16488_gb300 import ppsp
from workloads import CSRGraph, clique_pairs, csr_from_undirected, grid_graph, random_pairs, road_like_graph

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def road():
    import __graft_entry__

    __graft_entry__.build()
    g = road_like_graph(700, seed=61)
    with ppsp.Graph.from_csr(g) as G:
        yield g, G


def shape_of(G, pairs, **kw):
    with G.plan(pairs, **kw) as p:
        return p.launch_shape()


@pytest.mark.parametrize("mode", ["et", "bids", "bidastar"])
def test_one_group_at_a_time_gets_whole_ctas(road, mode):
    g, G = road
    pairs = random_pairs(g, 700, 62)
    few, many = (shape_of(G, pairs[:k], mode=mode, strategy="plain") for k in (10, 700))
    assert many["block_threads"] == 1024 and many["cluster"] == few["cluster"], (few, many)
    lane = shape_of(G, pairs, mode=mode, strategy="plain_star", max_ctas=19)
    assert lane["block_threads"] == 1024 and lane["ctas"] <= 19, lane


def test_team_of_one_cta_is_one_cta(road):
    g, G = road
    pairs = random_pairs(g, 400, 63)
    auto = shape_of(G, pairs[:6], mode="et", strategy="plain_star")
    assert auto["kernel"] == "clusters"
    for mode in ("et", "bids", "bidastar"):
        for k, strategy in ((6, "plain_star"), (6, "plain"), (400, "plain_star")):
            s = shape_of(G, pairs[:k], mode=mode, strategy=strategy, team_ctas=1)
            assert s["cluster"] == 1 and s["long_groups"] == 0 and s["ctas"] == s["teams"], (mode, k, s)


def test_clusters_of_512_threads(road):
    g, G = road
    pairs = random_pairs(g, 6, 64)
    want = oracle.pairs(g.offsets, g.targets, g.weights, pairs)
    for bits in (32, 64):
        s = shape_of(G, pairs, mode="et", strategy="plain_star", block_threads=512, dist_bits=bits)
        assert s["kernel"] == "clusters" and s["block_threads"] == 512, s
        got = G.batch(pairs, mode="et", strategy="plain_star", block_threads=512, dist_bits=bits)
        assert np.array_equal(got, want)


def test_ctas_of_256_threads(road):
    g, G = road
    pairs = random_pairs(g, 24, 76)
    want = oracle.pairs(g.offsets, g.targets, g.weights, pairs)
    for mode, kernel in (("bids", "general"), ("et", "general"), ("bidastar", "bucket"), ("astar", "bucket")):
        for k, strategy in ((24, "plain_star"), (1, "plain")):
            s = shape_of(G, pairs[:k], mode=mode, strategy=strategy, block_threads=256)
            assert (s["kernel"], s["block_threads"]) == (kernel, 256), (mode, s)
        assert np.array_equal(G.batch(pairs, mode=mode, strategy="plain_star", block_threads=256), want), mode


def test_fewer_teams_where_memory_is_short():
    g = road_like_graph(900, seed=65)
    pairs = random_pairs(g, 900, 66)
    want = oracle.pairs(g.offsets, g.targets, g.weights, pairs[:30])
    with ppsp.Graph.from_csr(g) as G:
        per = G.slot_bytes(2, 32)
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info()[0]
        for room in (40, 170):  # slots that fit beside the caller's tensors
            held = torch.empty(free - room * per - (64 << 20), dtype=torch.uint8, device="cuda")
            try:
                for mode in ("bids", "bidastar"):
                    got = G.batch(pairs, mode=mode, strategy="plain_star")
                    assert np.array_equal(got[:30], want), mode
            finally:
                del held
                torch.cuda.empty_cache()


@pytest.mark.parametrize("side", [64, 128, 256, 512])
def test_slots_in_proportion_to_the_graph(side):
    g = grid_graph(side, seed=67)
    with ppsp.Graph.from_csr(g) as G:
        assert G.slot_bytes(2, 32) <= 40 * 2 * g.n and G.slot_bytes(2, 64) <= 60 * 2 * g.n
        pairs = random_pairs(g, 300, 68)
        want = oracle.pairs(g.offsets, g.targets, g.weights, pairs)
        for delta in (0, 5000, 1 << 40):  # coarse increments overflow the buckets
            got = G.batch(pairs, mode="et", strategy="plain_star", delta=delta, team_ctas=1)
            assert np.array_equal(got, want), delta


def test_host_calls_do_not_wait_for_other_streams():
    g = grid_graph(64, seed=74)
    pair = random_pairs(g, 1, 75)
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    with ppsp.Graph.from_csr(g) as G, ppsp.Graph.from_csr(g) as H:
        # the search memory of one team is there (its first allocation is not the question)
        with G.plan(pair, mode="bids", strategy="plain_star", stream=mine.cuda_stream) as p:
            p.run(torch.zeros(1, dtype=torch.int64, device="cuda").data_ptr())
            p.sync()
        want = G.query(*pair[0].tolist())
        H.query(*pair[0].tolist())
        done = torch.cuda.Event()
        with torch.cuda.stream(other):
            torch.cuda._sleep(4_000_000_000)  # about two seconds
        done.record(other)
        for k in (1, 2000, 20000, 100000, 400000, 1):
            got = G.batch(np.tile(pair, (k, 1)), mode="bids", strategy="plain_star", stream=mine.cuda_stream)
            assert got.shape == (k,) and (got == want).all()
            assert not done.query(), f"the call with {k} pairs waited for another stream"
        done.synchronize()


@pytest.mark.parametrize("limit", [1 << 8, 1 << 10])
def test_spin_limit_counts_from_a_search_s_last_step(road, limit):
    g, G = road
    pairs = clique_pairs(g, 8, 73)
    want = oracle.pairs(g.offsets, g.targets, g.weights, pairs)
    assert shape_of(G, pairs, mode="bids", strategy="multi")["kernel"] == "bucket_teams"
    for _ in range(3):
        assert np.array_equal(G.batch(pairs, mode="bids", strategy="multi", spin_limit=limit), want)


def test_astar_increment_where_paths_have_few_hops():
    rng = np.random.default_rng(71)
    n = 1 << 17
    u, v = rng.integers(0, n, (2, 5 * n // 2))
    lo, hi = np.minimum(u, v), np.maximum(u, v)
    key = np.unique((lo * n + hi)[lo != hi])
    lo, hi = key // n, key % n
    xy = rng.uniform(0, 1000, (n, 2)).astype(np.float32)
    w = (10 * np.sqrt(((xy[lo].astype(float) - xy[hi]) ** 2).sum(1)) + rng.integers(10, 1000, lo.size)).astype(np.uint32)
    off, tgt, wt = csr_from_undirected(n, lo, hi, w)
    g = CSRGraph(n=n, offsets=off, targets=tgt, weights=wt, coords=xy,
                 lcc=np.flatnonzero(np.diff(off.astype(np.int64)) >= 2).astype(np.uint32))
    pairs = random_pairs(g, 8, 72)
    want = oracle.pairs(g.offsets, g.targets, g.weights, pairs)
    with ppsp.Graph.from_csr(g) as G:
        mean = int(round(G.info()["w_mean"]))
        for mode in ("astar", "bidastar"):
            got, auto = G.batch(pairs, mode=mode, strategy="plain_star", return_counters=True)
            _, one = G.batch(pairs, mode=mode, strategy="plain_star", delta=mean, return_counters=True)
            assert np.array_equal(got, want) and auto["rounds"] < 1.5 * one["rounds"], (mode, auto, one)


def test_estimates_without_a_scaled_potential():
    # one edge of weight 0 leaves no positive potential: lengths are not known
    g = road_like_graph(700, seed=69)
    u = np.repeat(np.arange(g.n), np.diff(g.offsets.astype(np.int64)))
    w = g.weights.copy()
    a, b = int(u[0]), int(g.targets[0])
    w[((u == a) & (g.targets == b)) | ((u == b) & (g.targets == a))] = 0
    pairs = random_pairs(g, 6, 70)
    want = oracle.pairs(g.offsets, g.targets, w, pairs)
    with ppsp.Graph(g.offsets, g.targets, w, g.coords) as G:
        assert G.info()["potential_scale"] == 0.0
        for mode in ("et", "astar"):
            assert shape_of(G, pairs, mode=mode, strategy="plain_star")["kernel"] == "clusters", mode
            assert np.array_equal(G.batch(pairs, mode=mode, strategy="plain_star"), want), mode
