"""Batches whose few longest groups run on more threads each, in a launch
beside the rest's: single CTAs and clusters for them, one and two groups per SM
for the rest, repeated runs, replay from a CUDA graph, and paths."""

import numpy as np
import pytest
import torch

import oracle
from paper_2506_16488_gb300 import ppsp
from workloads import random_pairs, road_like_graph

pytestmark = pytest.mark.gpu

SIDE = 300


@pytest.fixture(scope="module")
def road():
    import __graft_entry__

    __graft_entry__.build()
    g = road_like_graph(SIDE, seed=71)
    with ppsp.Graph.from_csr(g) as G:
        yield g, G


def mixed_pairs(g, near, far, seed):
    """`near` pairs a few vertices apart and `far` ones across the graph."""
    rng = np.random.default_rng(seed)
    xy = g.coords[g.lcc]
    order = np.lexsort((xy[:, 0], np.round(xy[:, 1], 0)))
    ids = g.lcc[order]
    a = rng.integers(0, len(ids) - 5, near)
    lo = g.lcc[np.argsort(xy.sum(1))]
    pairs = np.concatenate([np.stack([ids[a], ids[a + rng.integers(1, 5, near)]], 1),
                            np.stack([rng.choice(lo[:200], far), rng.choice(lo[-200:], far)], 1)])
    pairs = pairs[rng.permutation(len(pairs))].astype(np.uint32)
    return pairs, oracle.pairs(g.offsets, g.targets, g.weights, pairs)


# (near, far, groups per SM of the rest)
SHAPES = [(200, 1, 1), (500, 12, 1), (700, 1, 2), (900, 40, 2)]


@pytest.mark.parametrize("near,far,per_sm", SHAPES)
@pytest.mark.parametrize("mode,bits", [("bids", 32), ("bidastar", 32), ("bidastar", 64), ("et", 32), ("astar", 64)])
def test_long_groups_beside_the_rest(road, near, far, per_sm, mode, bits):
    g, G = road
    pairs, want = mixed_pairs(g, near, far, seed=near + far)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    out = torch.zeros(len(pairs), dtype=torch.int64, device="cuda")
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    teams = []
    for kw in ({}, {"stream": stream.cuda_stream}, {"stream": stream.cuda_stream, "cuda_graph": True},
               {"ring_entries": 2}):
        p = G.plan(pairs, mode=mode, strategy="plain_star", dist_bits=bits, **kw)
        teams.append(p.device_bytes()["teams"])
        for _ in range(3):
            out.zero_()
            torch.cuda.synchronize()
            p.run(out.data_ptr())
            p.sync()
            assert np.array_equal(out.cpu().numpy().astype(np.uint64), want), kw
        if "cuda_graph" in kw:
            assert p.uses_graph()
        p.close()
    if mode == "bidastar" and per_sm == 2:  # the estimates favour teams of their own
        assert min(teams) > per_sm * sms, teams
    assert np.array_equal(G.batch(pairs, mode=mode, strategy="plain_star", dist_bits=bits), want)


@pytest.mark.parametrize("near,far", [(700, 2), (300, 2)])
def test_long_groups_with_paths(road, near, far):
    g, G = road
    pairs, want = mixed_pairs(g, near, far, seed=5)
    st, d, paths, _ = G.batch_paths(pairs, 3000, mode="bidastar", strategy="plain_star")
    assert st == ppsp.OK and np.array_equal(d, want)
    for q in range(0, len(pairs), 7):
        path = paths[q]
        assert path[0] == pairs[q, 0] and path[-1] == pairs[q, 1]
        assert oracle.path_weight(g.offsets, g.targets, g.weights, path) == int(want[q])


@pytest.mark.parametrize("bits", [32, 64])
def test_long_groups_on_clusters(bits):
    """Steps large enough for clusters of CTAs to take the longest groups."""
    g = road_like_graph(2048, seed=72)
    pairs = random_pairs(g, 200, seed=6)
    want = oracle.pairs(g.offsets, g.targets, g.weights, pairs)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    with ppsp.Graph.from_csr(g) as G:
        out = torch.zeros(len(pairs), dtype=torch.int64, device="cuda")
        with G.plan(pairs, mode="bidastar", strategy="plain_star", dist_bits=bits) as p:
            assert p.device_bytes()["teams"] > sms
            for _ in range(2):
                p.run(out.data_ptr())
                p.sync()
                assert np.array_equal(out.cpu().numpy().astype(np.uint64), want)
        assert np.array_equal(G.batch(pairs, mode="bidastar", strategy="plain_star", dist_bits=bits), want)
