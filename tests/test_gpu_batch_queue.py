"""Batches whose small graphs are refined together in one persistent launch
(many of them on few workers): every graph bit-exact with the oracle, and which
way a batch takes.  The launch spares each graph the allocations of its own
refinement, so the number of allocations tells the ways apart."""
import numpy as np
import pytest
import torch

import graphgen
import oracle

pytestmark = pytest.mark.gpu

jet = pytest.importorskip("paper_2304_13194_gb300")


def _items(gs, ks):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    dev = [[torch.from_numpy(a).cuda() for a in (g.xadj, g.adjncy, g.vwgt, g.adjwgt)] for g in gs]
    return [dict(xadj=t[0], adjncy=t[1], vwgt=t[2], adjwgt=t[3], k=k, eps=0.03, seed=i + 3)
            for i, (t, k) in enumerate(zip(dev, ks))]


def _check(out, gs, ks):
    for i, ((part, cut, status, ms), g, k) in enumerate(zip(out, gs, ks)):
        ref = oracle.partition(g, k, 0.03, i + 3)
        assert status == ref.status and cut == ref.cut and ms > 0, i
        assert (part.cpu().numpy() == ref.part).all(), i


def _allocations(f):
    a0 = jet.binding.alloc_count()
    r = f()
    return r, jet.binding.alloc_count() - a0


def _small(count, lo, hi, seed):
    r = np.random.default_rng(seed)
    gs = [graphgen.rgg(int(n), seed=seed + i) for i, n in enumerate(r.integers(lo, hi, count - 4))]
    return gs + [graphgen.grid3d(12, 10, 9, vw=(1, 4), ew=(1, 10), seed=3), graphgen.grid2d(64, 64),
                 graphgen.rmat(11, seed=8, vw=(1, 3), ew=(1, 5)), graphgen.gnp(500, 0.2, seed=4, ew=(1, 9))]


# (graphs, parts, workers, options, whether the small graphs go into one launch)
WAYS = [
    ("20_graphs_1_worker", 20, [2, 8, 33, 64], 1, {}, True),
    ("20_graphs_2_workers", 20, [2, 8, 33, 64], 2, {}, False),
    ("many_parts_1_worker", 8, [256], 1, {}, True),
    ("no_resident_loop_2_workers", 8, [600], 2, {}, True),
    ("no_resident_loop_8_workers", 8, [600], 8, {}, False),
    ("two_blocks", 20, [16], 1, {"cluster_blocks": 2}, True),
    ("sixteen_blocks", 20, [16], 1, {"cluster_blocks": 16}, True),
    ("threshold_0", 20, [16], 1, {"cluster_max_n": 0}, False),
    ("host_loop", 20, [16], 1, {"flags": jet.FLAG_HOSTLOOP}, False),
]


@pytest.mark.parametrize("name,count,ks,workers,opts,queued", WAYS, ids=[w[0] for w in WAYS])
def test_small_graphs_of_a_batch(name, count, ks, workers, opts, queued):
    gs = _small(count, 700, 4097, 5)
    ks = [ks[i % len(ks)] for i in range(count)]
    items = _items(gs, ks)
    with jet.Context(0, **opts) as c:
        singly = 0
        for it in items:
            _, a = _allocations(lambda: c.partition(it["xadj"], it["adjncy"], it["vwgt"], it["adjwgt"], k=it["k"],
                                                    seed=it["seed"]))
            singly += a
        out, a = _allocations(lambda: c.partition_batch(items, workers=workers))
    _check(out, gs, ks)
    assert (a < singly) == queued      # otherwise the same ones, and one per worker


def test_queue_beside_larger_graphs_and_a_refused_one():
    """Larger graphs are partitioned by the workers in the same call; a graph
    over the weight limit gets its status and spoils no other."""
    gs = _small(20, 700, 4000, 9) + [graphgen.rgg(20000, seed=5), graphgen.grid3d(18, 17, 16, vw=(1, 4), ew=(1, 10), seed=1)]
    ks = [8 if i < 20 else 32 for i in range(len(gs))]
    items = _items(gs, ks)
    with jet.Context(0) as c:
        _check(c.partition_batch(items, workers=1), gs, ks)
        bad = [dict(it) for it in items]
        bad[3]["vwgt"] = torch.full_like(bad[3]["vwgt"], 2 ** 30)
        with pytest.raises(jet.JetError) as ei:
            c.partition_batch(bad, workers=1)
        assert ei.value.status == -6
        _check(c.partition_batch(items, workers=1), gs, ks)


def test_every_allocation_failure_in_a_queued_batch():
    gs = [graphgen.rgg(1300 + 50 * i, seed=i + 1) for i in range(4)]
    ks = [600] * 4
    items = _items(gs, ks)
    with jet.Context(0) as c:
        _, n = _allocations(lambda: _check(c.partition_batch(items, workers=1), gs, ks))
        try:
            for nth in range(1, n + 1):
                jet.binding.debug_fail_alloc(nth)
                with pytest.raises(jet.JetError) as ei:
                    c.partition_batch(items, workers=1)
                assert ei.value.status == -3, nth
                if nth % 8 == 0:
                    _check(c.partition_batch(items, workers=1), gs, ks)
        finally:
            jet.binding.debug_fail_alloc(0)
        _check(c.partition_batch(items, workers=1), gs, ks)
