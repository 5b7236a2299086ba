"""The resident level loop (a level kept in a cluster's shared memory) against
the CUDA-graph loop: the same trajectory at the sizes where its layout changes
— single vertices, slices with a remainder, blocks without vertices, one and
two bytes per part, rows for a thread, a warp and a block, more parts around a
vertex than a thread keeps, and the largest levels that fit."""
import numpy as np
import pytest
import torch

import graphgen
from helpers import graph_from_triples

pytestmark = pytest.mark.gpu

jet = pytest.importorskip("paper_2304_13194_gb300")


def _star(n, hubs, seed):
    """Ring of n vertices with `hubs` vertices joined to many others (rows past every length class)."""
    r = np.random.default_rng(seed)
    tri = [[v, (v + 1) % n, 2] for v in range(n)]
    seen = {tuple(sorted(t[:2])) for t in tri}
    for h in range(hubs):
        for u in r.choice(n, min(n - 1, 60 * (h + 1) ** 3), replace=False):
            e = tuple(sorted((h * 7 % n, int(u))))
            if e[0] != e[1] and e not in seen:
                seen.add(e)
                tri.append([*e, int(r.integers(1, 6))])
    return graph_from_triples(n, tri)


CASES = [
    ("one_vertex", lambda: graphgen.grid2d(1, 1), True, 2, {}),
    ("n33_k3", lambda: graphgen.grid2d(11, 3), True, 3, {}),
    ("n511_k64_w", lambda: graphgen.grid2d(73, 7, vw=(1, 4), ew=(1, 10), seed=2), False, 64, {}),
    ("n513_blocks2", lambda: graphgen.rgg(513, seed=3), True, 16, {"cluster_blocks": 2}),
    ("n8193_k255_w", lambda: graphgen.rgg(8193, seed=4, vw=(1, 4), ew=(1, 10)), False, 255, {}),
    ("n8193_k256", lambda: graphgen.rgg(8193, seed=5), True, 256, {}),
    ("n8193_k257", lambda: graphgen.rgg(8193, seed=6), True, 257, {}),
    ("star_rows", lambda: _star(6000, 4, 7), False, 24, {}),
    ("star_rows_blocks4", lambda: _star(6000, 4, 8), False, 5, {"cluster_blocks": 4, "hub_degree": 64}),
    ("dense_many_parts", lambda: graphgen.gnp(900, 0.05, seed=9, ew=(1, 9)), False, 40, {}),
    ("largest_k64_w", lambda: graphgen.grid3d(40, 38, 38, vw=(1, 4), ew=(1, 10), seed=10), False, 64, {}),
    ("largest_k8", lambda: graphgen.grid2d(253, 258), True, 8, {}),
]


@pytest.mark.parametrize("name,make,unit,k,opts", CASES, ids=[c[0] for c in CASES])
def test_resident_loop_equals_graph_loop(name, make, unit, k, opts):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    g = make()
    vw, ew = (None, None) if unit else (g.vwgt, g.adjwgt)
    r = np.random.default_rng(k)
    # slabs of uneven weight with misplaced vertices: Jetlp, Jetrw and Jetrs iterations
    part0 = np.minimum((k * (np.arange(g.n) / g.n) ** 1.3).astype(np.int32), k - 1)
    part0 = np.where(r.random(g.n) < 0.1, r.integers(0, k, g.n), part0).astype(np.int32)
    with jet.Context(0, **opts) as a, jet.Context(0, cluster_max_n=0) as b:
        for fine in (True, False):
            pa, ca = a.refine(g.xadj, g.adjncy, vw, ew, k, part0, seed=3, is_finest=fine)
            ta = a.last_trace()
            pb, cb = b.refine(g.xadj, g.adjncy, vw, ew, k, part0, seed=3, is_finest=fine)
            tb = b.last_trace()
            assert ca == cb and torch.equal(pa, pb) and a.last_status == b.last_status
            assert ta["iters"] == tb["iters"]
            assert all((ta[key] == tb[key]).all() for key in ("kind", "nx", "nm", "cut", "maxw"))


def test_statistics_equal_the_graph_loops():
    """Per level and kernel the byte model counts the same passes in both loops
    (the rebalancing tiles aside, whose size is the loop's own)."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    g = graphgen.grid3d(20, 20, 20, vw=(1, 4), ew=(1, 10), seed=3)
    rows = {}
    for name, opts in (("resident", {}), ("graph", {"cluster_max_n": 0})):
        with jet.Context(0, **opts) as c:
            _, _, st = c.partition(g.xadj, g.adjncy, g.vwgt, g.adjwgt, k=32, seed=1, return_stats=True)
        rows[name] = st
    a, b = rows["resident"], rows["graph"]
    names = jet.kernel_names()
    same = [names.index(x) for x in ("k_lp_scan", "k_lp_select", "k_afterburn", "k_apply", "k_rb_scan", "k_rb_cand")]
    assert all(x > 0 for x in a.cluster_blocks) and all(x == 0 for x in b.cluster_blocks)
    assert a.iters_lp == b.iters_lp and a.iters_rw == b.iters_rw and a.iters_rs == b.iters_rs
    assert a.cut_level == b.cut_level and all(t > 0 for t in a.ms_level)
    for la, lb in zip(a.kern_bytes, b.kern_bytes):
        assert [la[i] for i in same] == [lb[i] for i in same]
