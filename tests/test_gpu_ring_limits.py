"""Rings whose 64-bit buckets would not fit shared memory: the plan keeps its
kernel with the largest ring that fits."""

import numpy as np
import pytest

import oracle
from paper_2506_16488_gb300 import ppsp
from workloads import random_pairs, road_like_graph

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ring", [223, 224, 256])
@pytest.mark.parametrize("bits", [32, 64])
def test_large_rings(ring, bits):
    g = road_like_graph(400, seed=91)
    pairs = random_pairs(g, 400, 92)
    want = oracle.pairs(g.offsets, g.targets, g.weights, pairs)
    with ppsp.Graph.from_csr(g) as G:
        for mode in ("bids", "bidastar", "et"):
            for k, strategy in ((1, "plain"), (8, "plain_star"), (400, "plain_star")):
                shapes = []
                for r in (0, ring):
                    with G.plan(pairs[:k], mode=mode, strategy=strategy, dist_bits=bits, ring_entries=r) as p:
                        shapes.append(p.launch_shape()["kernel"])
                assert shapes[0] == shapes[1] != "general", (mode, k, shapes)
                got = G.batch(pairs[:k], mode=mode, strategy=strategy, dist_bits=bits, ring_entries=ring)
                assert np.array_equal(got, want[:k]), (mode, k)
            assert G.query(*pairs[3].tolist(), mode=mode, dist_bits=bits, ring_entries=ring) == int(want[3])
