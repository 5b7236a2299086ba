"""Which loop refines a level: the resident loop (a cluster that keeps the level
in its shared memory), the cluster loop on the level's state in global memory,
or the CUDA-graph loop; and that all of them give the same result.  One level
per call (max_levels=1)."""
import numpy as np
import pytest
import torch

import graphgen

pytestmark = pytest.mark.gpu

jet = pytest.importorskip("paper_2304_13194_gb300")


def _dev(g, unit):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    one = np.ones(g.n, np.int32)      # given, so that no call allocates unit weights
    return [torch.from_numpy(a).cuda() if a is not None else None
            for a in (g.xadj, g.adjncy, one if unit else g.vwgt, None if unit else g.adjwgt)]


@pytest.mark.parametrize("chosen,expect", [(None, False), (5999, False), (6000, True), (1 << 20, True)],
                         ids=["default", "below", "equal", "above"])
def test_chosen_cluster_max_n_holds_for_levels_that_do_not_fit(chosen, expect):
    """600 parts do not fit the resident loop: 6,000 vertices take the cluster
    loop when the caller's cluster_max_n allows them, and only then."""
    g, k = graphgen.rgg(6000, seed=4, vw=(1, 4), ew=(1, 10)), 600
    t = _dev(g, False)
    opts = {} if chosen is None else {"cluster_max_n": chosen}
    with jet.Context(0, max_levels=1, **opts) as c:
        part, cut, st = c.partition(*t, k=k, seed=2, return_stats=True)
    assert (st.cluster_blocks[0] > 0) == expect
    with jet.Context(0, max_levels=1, cluster_max_n=0) as c:
        ref, ref_cut, st = c.partition(*t, k=k, seed=2, return_stats=True)
    assert st.cluster_blocks[0] == 0 and cut == ref_cut and torch.equal(part, ref)


def _start(g, k):
    """Slabs of uneven weight with misplaced vertices: Jetlp, Jetrw and Jetrs iterations."""
    r = np.random.default_rng(k)
    part = np.minimum((k * (np.arange(g.n) / g.n) ** 1.3).astype(np.int32), k - 1)
    return np.where(r.random(g.n) < 0.1, r.integers(0, k, g.n), part).astype(np.int32)


def _random_graph(n, entries, seed):
    """Uniform random weighted graph of n vertices and about `entries` CSR entries (no locality)."""
    r = np.random.default_rng(seed)
    u, v = r.integers(0, n, (2, entries // 2))
    a, b = np.minimum(u, v)[u != v], np.maximum(u, v)[u != v]
    key = np.unique(a.astype(np.int64) * n + b)
    a, b = key // n, key % n
    w = r.integers(1, 11, len(key)).astype(np.int32)
    src, dst, ww = np.concatenate([a, b]), np.concatenate([b, a]), np.concatenate([w, w])
    o = np.lexsort((dst, src))
    xadj = np.zeros(n + 1, np.int64)
    xadj[1:] = np.cumsum(np.bincount(src, minlength=n))
    return graphgen.Graph(n, xadj, dst[o].astype(np.int32), r.integers(1, 5, n).astype(np.int32), ww[o], "random")


# (vertices, entries, parts, whether a cluster refines the level): both sides of the line at each size class
LINE = [
    (40000, 440000, 8, True), (40000, 480000, 8, False), (40000, 320000, 64, True), (40000, 360000, 64, False),
    (20000, 170000, 256, True), (20000, 200000, 256, False), (32768, 880000, 256, False),
    (7000, 330000, 16, True), (7000, 365000, 16, False), (7000, 70000, 256, True), (7000, 85000, 256, False),
]


@pytest.mark.parametrize("n,entries,k,cluster", LINE)
def test_levels_of_many_entries_leave_the_resident_loop(n, entries, k, cluster):
    g = _random_graph(n, entries, n + k)
    t = _dev(g, False)
    with jet.Context(0, max_levels=1) as a, jet.Context(0, max_levels=1, cluster_max_n=0) as b:
        st = a.partition(*t, k=k, seed=2, return_stats=True)[2]
        assert (st.cluster_blocks[0] > 0) == cluster
        part = torch.from_numpy(_start(g, k)).cuda()
        for fine in (True, False):
            pa, ca = a.refine(*t, k, part, seed=3, is_finest=fine)
            ta = a.last_trace()
            pb, cb = b.refine(*t, k, part, seed=3, is_finest=fine)
            tb = b.last_trace()
            assert ca == cb and a.last_status == b.last_status and torch.equal(pa, pb)
            assert ta["iters"] == tb["iters"]
            assert all((ta[key] == tb[key]).all() for key in ("kind", "nx", "nm", "cut", "maxw"))
