"""The byte model of the kernels that mark and list moves, against its formulas
over the iteration record: a marked move is 8 bytes, its list entry 4, and what
a kernel reads to make them is counted once."""
import numpy as np
import pytest
import torch

import graphgen
import oracle

pytestmark = pytest.mark.gpu

jet = pytest.importorskip("paper_2304_13194_gb300")

TILE = 256                                  # vertices per rebalancing tile of the CUDA-graph loop
LOOPS = {"graph": {"cluster_max_n": 0}, "resident": {}}


def _run(g, k, eps, **opts):
    """(bytes per kernel, iteration record, partition's start cut) of a one-level partition."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    with jet.Context(0, max_levels=1, **opts) as c:
        _, _, st = c.partition(g.xadj, g.adjncy, g.vwgt, g.adjwgt, k=k, eps=eps, seed=2, return_stats=True)
        return dict(zip(jet.kernel_names(), st.kern_bytes[0])), c.last_trace(), st


@pytest.mark.parametrize("loop", LOOPS)
def test_bytes_of_the_moves_without_an_afterburner(loop):
    g, k, eps = graphgen.grid3d(18, 17, 16, vw=(1, 4), ew=(1, 10), seed=3), 16, 1.0
    b, tr, _ = _run(g, k, eps, flags=jet.FLAG_NO_AFTERBURN, **LOOPS[loop])
    assert (tr["kind"] == jet.KIND_LP).all() and tr["nm"].sum() > 0
    best, copies = oracle.cut(g, oracle.initial_partition(g, k)), 0
    for i, cut in enumerate(tr["cut"]):     # P_best is copied in the iteration after an improvement
        if cut < best:
            best = cut
            copies += i + 1 < tr["iters"]
    assert b["k_afterburn"] == int((4 * tr["nx"] + 16 * tr["nm"]).sum()) + 8 * g.n * copies


@pytest.mark.parametrize("weak_limit", [0, 1000], ids=["strong", "weak"])
@pytest.mark.parametrize("loop", LOOPS)
def test_bytes_of_the_rebalancing_moves(loop, weak_limit):
    g, k = graphgen.grid3d(18, 17, 16, vw=(1, 4), ew=(1, 10), seed=3), 16
    b, tr, _ = _run(g, k, 0.0, weak_limit=weak_limit, **LOOPS[loop])
    rw, rs = tr["kind"] == jet.KIND_RW, tr["kind"] == jet.KIND_RS
    assert (rs if weak_limit == 0 else rw).any() and tr["nm"][rw | rs].sum() > 0
    n, tiles = g.n, -(-g.n // TILE) if loop == "graph" else 0
    c, m = tr["nx"], tr["nm"]
    if loop == "graph":
        assert b["k_rb_tilescan"] > 0
        assert b["k_rb_tilehist"] == int((4 * n + 4 * c)[rw | rs].sum()) + b["k_rb_tilescan"] // 2
    else:                                   # no tiles there, and no kernels over them
        assert b["k_rb_tilescan"] == 0 and b["k_rb_tilehist"] == 0
    assert b["k_rb_take"] == int((4 * n + 4 * c + 16 * m)[rw].sum() + (12 * n + 8 * tiles + 4 * c)[rs].sum()) + \
        b["k_rb_tilescan"] // 2
    assert b["k_rb_cookie"] == int((8 * n + 8 * tiles + 20 * m)[rs].sum())
