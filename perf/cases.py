"""Performance cases: the calls a program that uses this library makes, with
the graphs, batches and options it makes them with.

A program loads a graph once, keeps the handle (and, with BiDS or BiD-A*, the
stepping-increment model attached to it) and then asks for distances: one
query at a time, batches of pairs, batches with paths, or a prepared plan it
replays.  So a case's graph depends on the case alone and is kept between
states, and the queries come from the seed.  Graphs are the library's own
recipes, generated on the GPU: jittered grids, road-like grids (10% of the
grid edges deleted, 0.5% short shortcuts), one-way variants of them, and
power-law RMAT graphs (edge factor 16).

A case is a dict of
  graph     "grid", "road" or "rmat"
  size      side of the grid, or the RMAT scale
  unit      weight of a unit-length edge of a road-like graph (1000, or 20000
            where paths are compared: then no two shortest paths are equally
            long)
  oneway    30% of the edges keep one direction only (a directed graph)
  shape     "random" pairs, "tercile" (near / mid / far by grid distance),
            "clique" or "star" query graphs, "roadmix" (random pairs and a
            32-clique), "socialmix" (random pairs, a 64-leaf star and an
            11-clique)
  k         number of queries
  mode, strategy, bits   plug-in, batch strategy and distance width
  entry     "query" (Graph.query), "batch" (Graph.batch), "paths"
            (Graph.batch_paths) or "plan" (Plan.run into a device buffer)
"""

import math

import numpy as np
import torch

from paper_2506_16488_gb300 import learned_delta, ppsp

DEV = "cuda"


def _case(name, graph, size, shape, k, mode, strategy="auto", entry="batch", bits=32, oneway=False, unit=1000):
    c = {"graph": graph, "size": size, "shape": shape, "k": k, "mode": mode, "strategy": strategy,
         "entry": entry, "bits": bits, "oneway": oneway, "unit": unit}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one BiDS query on the smallest graph: the latency of a call
        _case("query_grid64", "grid", 64, "random", 1, "bids", "multi", "query"),
        # the small batch of the benchmark: 100 random pairs, BiDS, default strategy
        _case("batch_grid64", "grid", 64, "random", 100, "bids", "multi"),
        # one interactive route query on a city-sized road graph
        _case("query_road1024", "road", 1024, "random", 1, "bidastar", "multi", "query"),
        # a handful of route queries at once (a dispatcher's request): fewer queries than SMs
        _case("few_road1024", "road", 1024, "random", 16, "bidastar"),
        # the benchmark's 1,000 near / mid / far route queries
        _case("batch_road1024", "road", 1024, "tercile", 1000, "bidastar"),
        # a distance matrix: all pairs of 24 places, shared BiDS searches (Multi-BiDS)
        _case("clique_road1024", "road", 1024, "clique", 24, "bids", "multi"),
        # one-way streets (directed, odd size), one-directional A*
        _case("astar_oneway500", "road", 500, "random", 300, "astar", "auto", oneway=True),
        # routes with their vertices, BiDS, one group per query
        _case("paths_road512", "road", 512, "random", 64, "bids", "plain_star", "paths", unit=20000),
        # the benchmark's headline batch as a prepared plan into a device buffer
        _case("plan_road2048", "road", 2048, "roadmix", 2048, "bidastar", "auto", "plan"),
        # the largest road graph, uint64 distances, a serving batch of 256 pairs
        _case("batch_road4096_u64", "road", 4096, "random", 256, "bidastar", "auto", bits=64),
        # one BiDS query on a social-network-like graph
        _case("query_rmat20", "rmat", 20, "random", 1, "bids", "multi", "query"),
        # the benchmark's social batch (random pairs, a star and a clique), strategy chosen per component
        _case("batch_rmat20", "rmat", 20, "socialmix", 183, "bids", "auto"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["road", "road", "road", "grid", "rmat"])
    if kind == "rmat":
        scale = rng.randint(10, 20)
        entry = rng.choice(["query", "batch", "batch", "plan"])
        if entry == "query":
            return _case("", "rmat", min(scale, 19), "random", 1, "bids", "multi", entry, bits=rng.choice([32, 64]))
        shape = rng.choice(["random", "random", "star", "clique"])
        k = {"random": _log_int(rng, 2, 96), "star": _log_int(rng, 4, 64), "clique": rng.randint(3, 11)}[shape]
        # Multi-BiDS on large social graphs takes longer than any listed case
        strategy = "multi" if scale <= 16 and rng.random() < 0.5 else "auto"
        return _case("", "rmat", scale, shape, k, "bids", strategy, entry, bits=rng.choice([32, 32, 64]))
    size = _log_int(rng, 40, 400) if kind == "grid" else _log_int(rng, 100, 2048)
    mode = rng.choice(["bidastar", "bidastar", "bidastar", "bids", "bids", "astar", "et"])
    entry = rng.choice(["query", "batch", "batch", "batch", "plan", "paths"])
    oneway = kind == "road" and rng.random() < 0.2
    bits = rng.choice([32, 32, 32, 64])
    # settled area over all queries, against that of the listed batches
    cost = {"bidastar": 1, "bids": 6, "astar": 6, "et": 12}[mode] * size * size
    most = max(2, min(2048, int(4e9 / cost)))
    if entry == "query":
        return _case("", kind, size, "random", 1, mode, "multi", entry, bits, oneway)
    if entry == "paths":
        k = min(most, _log_int(rng, 2, 128))
        return _case("", kind, size, "random", k, mode, "plain_star", entry, bits, oneway, 20000)
    shape = rng.choice(["random", "random", "tercile", "clique", "star"])
    if shape == "clique":
        return _case("", kind, size, shape, rng.randint(3, max(3, min(24, int(math.sqrt(2 * most))))), mode,
                     "multi" if mode == "bids" and size <= 1024 else "auto", entry, bits, oneway)
    k = min(most, _log_int(rng, 4, 64) if shape == "star" else _log_int(rng, 2, 2048))
    return _case("", kind, size, shape, k, mode, "auto", entry, bits, oneway)


# ---- graphs ----------------------------------------------------------------
def _pairs_of(n, keys):
    """Both directions of the undirected edges lo * n + hi, sorted by row and
    target, and each one's edge number."""
    lo, hi = keys // n, keys % n
    both = torch.cat([lo * n + hi, hi * n + lo])
    both, order = torch.sort(both)
    return both // n, both % n, order % keys.numel()


def _csr(n, src, dst, w):
    off = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(torch.bincount(src, minlength=n), 0)
    return (off.cpu().numpy().astype(np.uint64), dst.cpu().numpy().astype(np.uint32),
            w.cpu().numpy().astype(np.uint32))


def _make_csr(case):
    """(offsets, targets, weights, coords or None, grid cells or None), host arrays."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(1000 * case["size"] + len(case["graph"]) + (7 if case["oneway"] else 0))

    def rand(*shape):
        return torch.rand(*shape, generator=gen, device=DEV)

    if case["graph"] == "rmat":
        scale, n = case["size"], 1 << case["size"]
        u = torch.zeros(16 * n, dtype=torch.int64, device=DEV)
        v = torch.zeros_like(u)
        for level in range(scale):  # quadrants with probabilities 0.57, 0.19, 0.19, 0.05
            r = rand(16 * n)
            u += (r >= 0.76).long() << level
            v += (((r >= 0.57) & (r < 0.76)) | (r >= 0.95)).long() << level
        keys = torch.unique((torch.minimum(u, v) * n + torch.maximum(u, v))[u != v])
        w = torch.randint(1, 65536, (keys.numel(),), generator=gen, device=DEV)
        src, dst, edge = _pairs_of(n, keys)
        return (*_csr(n, src, dst, w[edge]), None, None)

    side, n = case["size"], case["size"] ** 2
    ids = torch.arange(n, device=DEV)
    cell = torch.stack([ids % side, ids // side], 1)
    xy = (cell.double() + (rand(n, 2).double() - 0.5) * 0.6).float()
    grid = ids.view(side, side)
    keys = torch.cat([(grid[:, :-1] * n + grid[:, 1:]).reshape(-1), (grid[:-1] * n + grid[1:]).reshape(-1)])
    edges = keys.numel()
    if case["graph"] == "road":
        keys = keys[rand(edges) >= 0.1]
        short = max(1, edges // 200)  # shortcuts of at most 20 cells
        a = torch.randint(0, n, (4 * short,), generator=gen, device=DEV)
        d = torch.randint(-20, 21, (4 * short, 2), generator=gen, device=DEV)
        to = cell[a] + d
        fine = ((d * d).sum(1) <= 400) & (d != 0).any(1) & (to >= 0).all(1) & (to < side).all(1)
        a, b = a[fine][:short], (to[:, 1] * side + to[:, 0])[fine][:short]
        keys = torch.unique(torch.cat([keys, torch.minimum(a, b) * n + torch.maximum(a, b)]))
    else:
        keys = torch.sort(keys)[0]
    lo, hi = keys // n, keys % n
    length = (xy[lo].double() - xy[hi].double()).square().sum(1).sqrt()
    w = torch.round(case["unit"] * length).long().clamp_(min=1)
    if case["graph"] == "grid":
        w += torch.randint(0, 101, (keys.numel(),), generator=gen, device=DEV)
    src, dst, edge = _pairs_of(n, keys)
    w = w[edge]
    if case["oneway"]:
        way = rand(keys.numel())[edge]  # < 0.15: only upwards, 0.15 .. 0.3: only downwards
        keep = (way >= 0.3) | ((way < 0.15) == (src < dst))
        src, dst, w = src[keep], dst[keep], w[keep]
    return (*_csr(n, src, dst, w), xy.cpu().numpy(), cell.cpu().numpy())


class _Loaded:
    """A graph as a program keeps it: the handle with its models attached."""

    def __init__(self, case):
        off, tgt, w, xy, cell = _make_csr(case)
        torch.cuda.empty_cache()
        self.csr = (off, tgt, w)
        self.cell = cell
        self.graph = ppsp.Graph(off, tgt, w, xy, undirected=not case["oneway"])
        for mode in ("bids", "bidastar"):
            if mode == "bids" or xy is not None:
                self.graph.set_delta_model(mode, learned_delta.load_model(mode))
        # endpoints: any vertex that is no dead end
        self.pool = np.flatnonzero(np.diff(off.astype(np.int64)) >= 2)


_kept = {}  # the graph in use (at most one)


def _load(case):
    key = (case["graph"], case["size"], case["oneway"], case["unit"])
    if key not in _kept:
        _kept.clear()
        _kept[key] = _Loaded(case)
    return _kept[key]


def _queries(case, g, seed):
    rng = np.random.default_rng([seed, case["k"], case["size"]])
    pool, k = g.pool, case["k"]

    def rand(count):
        return pool[rng.integers(0, pool.size, (count, 2))]

    def clique(size):
        v = pool[rng.choice(pool.size, size, replace=False)]
        i, j = np.triu_indices(size, 1)
        return np.stack([v[i], v[j]], 1)

    def star(leaves):
        v = pool[rng.choice(pool.size, leaves + 1, replace=False)]
        return np.stack([np.full(leaves, v[0]), v[1:]], 1)

    shape = case["shape"]
    if shape == "random":
        p = rand(k)
    elif shape == "clique":  # k vertices
        p = clique(k)
    elif shape == "star":  # k leaves
        p = star(k)
    elif shape == "tercile":
        cand = rand(30 * k)
        order = np.argsort(np.abs(g.cell[cand[:, 0]] - g.cell[cand[:, 1]]).sum(1), kind="stable")
        sizes = [k // 3, k // 3, k - 2 * (k // 3)]
        parts = [rng.choice(order[10 * k * j:10 * k * (j + 1)], s, replace=False) for j, s in enumerate(sizes)]
        p = cand[np.concatenate(parts)]
    elif shape == "roadmix":  # 496 of the queries: every pair of a 32-clique
        p = np.concatenate([rand(k - 496), clique(32)])
    elif shape == "socialmix":  # a 64-leaf star and an 11-clique (55 pairs) among them
        p = np.concatenate([rand(k - 119), star(64), clique(11)])
    else:
        raise ValueError(shape)
    return np.ascontiguousarray(p, dtype=np.uint32)


# ---- the measured calls ----------------------------------------------------
class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = case
    s.loaded = _load(case)
    s.graph = s.loaded.graph
    s.pairs = _queries(case, s.loaded, seed)
    s.opts = {"mode": case["mode"], "dist_bits": case["bits"]}
    if case["entry"] == "query":
        s.s, s.t = (int(x) for x in s.pairs[0])
    else:
        s.opts["strategy"] = case["strategy"]
    if case["entry"] == "plan":
        s.plan = s.graph.plan(s.pairs, **s.opts)
        s.out = torch.zeros(s.pairs.shape[0], dtype=torch.int64, device=DEV)
    return s


def run(state):
    s = state
    entry = s.case["entry"]
    if entry == "query":
        d = s.graph.query(s.s, s.t, **s.opts)
        return -1 if d == ppsp.INF else d
    if entry == "plan":
        s.plan.run(s.out.data_ptr())
        return s.out  # uint64 distances, the unreachable ones all ones (-1)
    if entry == "paths":
        room = 6 * s.case["size"]  # vertices per path: more than the longest one has
        status, dist, paths, lens = s.graph.batch_paths(s.pairs, room, **s.opts)
        rows = np.full((len(paths), room), -1, dtype=np.int32)
        for row, path in zip(rows, paths):
            row[:path.size] = path
        return {"distances": dist.view(np.int64), "lengths": lens.view(np.int64), "paths": rows}
    return s.graph.batch(s.pairs, **s.opts).view(np.int64)


def _counts(case):
    """(vertices, adjacency entries, queries) of a case, to within a few per cent."""
    k = case["k"]
    if case["shape"] == "clique":
        k = k * (k - 1) // 2
    if case["graph"] == "rmat":
        return 1 << case["size"], 30 << case["size"], k
    side = case["size"]
    share = 1.0 if case["graph"] == "grid" else 0.905
    return side * side, int(share * 4 * side * (side - 1) * (0.85 if case["oneway"] else 1.0)), k


def work(case):
    """The graph read once (offsets, targets and weights, with A* the
    coordinates; a directed graph in both directions for a bidirectional
    mode), the pairs read and the answers written once; an addition and a
    comparison per adjacency entry."""
    n, m, k = _counts(case)
    b = 4 * (n + 1) + 8 * m
    if case["oneway"] and case["mode"].startswith("bid"):
        b *= 2
    if case["mode"].endswith("astar"):
        b += 8 * n
    return {"bytes": b + 16 * k, "flops": 2 * m}


def exact(case, seed):
    """Bellman-Ford over all queries at once, where it is quick."""
    n, m, k = _counts(case)
    if case["graph"] == "rmat" or case["entry"] == "paths" or m * k > 1 << 25:
        return None
    g = _load(case)
    pairs = _queries(case, g, seed)
    off, tgt, w = g.csr
    src = torch.from_numpy(np.repeat(np.arange(off.size - 1), np.diff(off.astype(np.int64)))).to(DEV)
    dst = torch.from_numpy(tgt.astype(np.int64)).to(DEV)
    wt = torch.from_numpy(w.astype(np.int64)).to(DEV)
    starts, row = np.unique(pairs[:, 0], return_inverse=True)
    far = 1 << 60
    d = torch.full((starts.size, off.size - 1), far, dtype=torch.int64, device=DEV)
    d[torch.arange(starts.size, device=DEV), torch.from_numpy(starts.astype(np.int64)).to(DEV)] = 0
    into = dst.expand(starts.size, -1)
    while True:
        new = d.scatter_reduce(1, into, d[:, src] + wt, "amin")
        if torch.equal(new, d):
            break
        d = new
    got = d.cpu().numpy()[row.reshape(-1), pairs[:, 1].astype(np.int64)]
    got = np.where(got >= far, -1, got)
    return int(got[0]) if case["entry"] == "query" else got
