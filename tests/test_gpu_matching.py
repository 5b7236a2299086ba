"""Heavy-edge matching against the oracle where its forms change: level sizes
around a warp's word, a block's slice and the largest one-cluster level, rows
around the short, warp and block lengths, equal and distinct weights, none at
all.  Matchings are whole numbers and must be the same."""
import numpy as np
import pytest
import torch

import graphgen
import oracle
from helpers import graph_from_triples

pytestmark = pytest.mark.gpu

jet = pytest.importorskip("paper_2304_13194_gb300")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    c = jet.Context(0)
    yield c
    c.close()


def _stars(*leaves, pairs=False):
    """A chain of hubs with the given numbers of leaves; with pairs, neighbouring
    leaves share a heavier edge, so that they match and the hubs' rows shrink."""
    t, hub = [], 0
    for i, m in enumerate(leaves):
        t += [[hub, hub + 1 + j, 1 + (j * 7) % 5] for j in range(m)]
        if pairs:
            t += [[hub + 1 + j, hub + 2 + j, 9] for j in range(0, m - 1, 2)]
        if i + 1 < len(leaves):
            t.append([hub, hub + m + 1, 3])
        hub += m + 1
    return graph_from_triples(hub, t)


CASES = [
    ("two", lambda: graph_from_triples(2, [[0, 1, 1]])),
    ("path33", lambda: graph_from_triples(33, [[i, i + 1, 1 + i % 3] for i in range(32)])),
    ("isolated", lambda: graphgen.gnp(1000, 0.0008, seed=1)),
    ("grid_w", lambda: graphgen.grid2d(127, 258, vw=(1, 3), ew=(1, 4), seed=2)),       # 32766: one cluster
    ("grid_limit", lambda: graphgen.grid2d(256, 128)),                                # 32768
    ("grid_over", lambda: graphgen.grid2d(32769, 1)),
    ("grid3d", lambda: graphgen.grid3d(30, 31, 32, ew=(1, 9), seed=4)),
    ("rmat_w", lambda: graphgen.rmat(13, seed=3, vw=(1, 2), ew=(1, 9))),
    ("rmat_large", lambda: graphgen.rmat(17, seed=5)),
    ("stars", lambda: _stars(15, 16, 17, 33, 511, 512, 513, 1023, 1025, 5000)),
    ("stars_cluster", lambda: _stars(*([2] * 5000), 16, 17, 33, 511, 512, 513, 1023, 1025, 5000)),
    ("stars_large", lambda: _stars(*([3] * 9000), 16, 17, 1024, 1025, 5000)),
]


@pytest.mark.parametrize("name,make", CASES, ids=[c[0] for c in CASES])
def test_matching_equals_oracle(ctx, name, make):
    g = make()
    d = [None if a is None else torch.as_tensor(np.asarray(a)).cuda() for a in (g.xadj, g.adjncy, g.adjwgt)]
    for weights in (d[2], None):
        for level, rounds in ((0, 8), (3, 1), (1, 0)):
            gw = g if weights is not None else graphgen.Graph(g.n, g.xadj, g.adjncy, g.vwgt, np.ones_like(g.adjncy))
            got = ctx.hem(d[0], d[1], weights, seed=11, level=level, rounds=rounds).cpu().numpy()
            assert np.array_equal(got, oracle.hem(gw, 11, level, rounds)), (weights is None, level, rounds)


HIERARCHIES = [
    ("path2048", lambda: graphgen.grid2d(2048, 1), 2),              # one scan tile
    ("path2049", lambda: graphgen.grid2d(2049, 1), 2),              # two
    ("path_scan_limit", lambda: graphgen.grid2d(2097152, 1), 512),  # 1,024 tiles: every tile adds up its own offset
    ("path_scan_over", lambda: graphgen.grid2d(2097153, 1), 512),   # 1,025: a scan of the sums
    ("no_match", lambda: graphgen.Graph(3000, np.zeros(3001, np.int64), np.zeros(0, np.int32), np.ones(3000, np.int32),
                                        np.zeros(0, np.int32)), 2),
    # merged rows around the thread, warp and block classes, the last one past the largest block row
    ("row_classes", lambda: _stars(*range(10, 20), *range(27, 35), *range(250, 260), *range(510, 514),
                                    *range(4088, 4100), 6000, pairs=True), 2),
    ("dense", lambda: graphgen.gnp(700, 0.9, seed=6, ew=(1, 9)), 2),
]


@pytest.mark.parametrize("name,make,k", HIERARCHIES, ids=[c[0] for c in HIERARCHIES])
def test_hierarchy_equals_oracle(ctx, name, make, k):
    g = make()
    ref = oracle.coarsen(g, k, seed=5)
    d = [torch.as_tensor(np.asarray(a)).cuda() for a in (g.xadj, g.adjncy, g.vwgt, g.adjwgt)]
    h = ctx.coarsen(*d, k=k, seed=5)
    try:
        assert h.info()[0] == len(ref)
        for i in range(len(ref)):
            L, R = h.level(i), ref[i].graph
            assert L["n"] == R.n
            for key, want in (("xadj", R.xadj), ("adjncy", R.adjncy), ("vwgt", R.vwgt), ("adjwgt", R.adjwgt)):
                assert np.array_equal(np.asarray(L[key].cpu()), want), (i, key)
            if i + 1 < len(ref):
                assert np.array_equal(np.asarray(L["cmap"].cpu()), ref[i].cmap), i
    finally:
        h.close()


def _splitmix64(x):
    x = np.asarray(x, np.uint64) + np.uint64(0x9E3779B97F4A7C15)
    x = (x ^ (x >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return x ^ (x >> np.uint64(31))


def _csr(n, pairs):
    return graph_from_triples(n, [[a, b, 1] for a, b in pairs])


def _colliding_twins():
    """Two groups of twins, interleaved by id, whose 64-bit neighbourhood hashes
    differ but share their low 24 bits (as many as 220 vertices are sorted by)."""
    hubs = 160
    h = _splitmix64(np.arange(hubs, dtype=np.uint64) ^ np.uint64(0x2545F4914F6CDD1D))
    a, b = np.triu_indices(hubs, 1)
    s = h[a] + h[b]
    low = s & np.uint64((1 << 24) - 1)
    order = np.argsort(low, kind="stable")
    hit = next(i for i in range(len(order) - 1)
               if low[order[i]] == low[order[i + 1]] and s[order[i]] != s[order[i + 1]])
    p, q = order[hit], order[hit + 1]
    pairs = [(i, i + 1) for i in range(0, hubs, 2)]
    for j in range(60):
        e = (p, q)[j % 3 == 1]
        pairs += [(int(a[e]), hubs + j), (int(b[e]), hubs + j)]
    mate = np.full(220, -1, np.int32)
    mate[:hubs] = np.arange(hubs) ^ 1
    return _csr(220, pairs), mate


def _two_hop_mix(n, seed):
    """n vertices, most of them leaves, twins and relatives of a few hubs."""
    r = np.random.default_rng(seed)
    hubs = max(2, n // 50)
    t = [(i, (i + 1) % hubs) for i in range(hubs if hubs > 2 else 1)]
    kind = r.integers(0, 3, n - hubs)
    x = r.integers(0, hubs, (n - hubs, 2))
    x[kind == 1] = (x[kind == 1] // 4) * 4 % hubs
    for i in range(n - hubs):
        t.append((int(x[i, 0]), hubs + i))
        if kind[i] and x[i, 0] != x[i, 1]:
            t.append((int(x[i, 1]), hubs + i))
    return _csr(n, t)


@pytest.mark.parametrize("n", [3, 31, 2047, 2049, 262144, 262145])
def test_two_hop_equals_oracle(ctx, n):
    g = _two_hop_mix(n, n)      # 262,144: the last size whose tiles add the histograms up
    mate = oracle.hem(g, 7, 0, 2)
    got, added = ctx.two_hop(torch.as_tensor(g.xadj).cuda(), torch.as_tensor(g.adjncy).cuda(), torch.as_tensor(mate).cuda())
    want, wadded = oracle.two_hop(g, mate)
    assert list(added) == wadded and np.array_equal(got.cpu().numpy(), want)


def test_twins_that_share_the_sorted_bits(ctx):
    g, mate = _colliding_twins()
    want, wadded = oracle.two_hop(g, mate)
    assert wadded[1] > 0
    got, added = ctx.two_hop(torch.as_tensor(g.xadj).cuda(), torch.as_tensor(g.adjncy).cuda(), torch.as_tensor(mate).cuda())
    assert list(added) == wadded and np.array_equal(got.cpu().numpy(), want)
