"""Rebalancing passes where the slot buckets change their place and their
sums are largest: one, 124 and 125 oversized parts (4,096 buckets are kept per
block, 33 per part) and vertex weights that add up to nearly 2^31, element by
element against the oracle."""
import numpy as np
import pytest
import torch

import graphgen
import oracle

pytestmark = pytest.mark.gpu

jet = pytest.importorskip("paper_2304_13194_gb300")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    c = jet.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("strong", [False, True])
@pytest.mark.parametrize("over", [1, 124, 125])
@pytest.mark.parametrize("vw", [1, 261000])
def test_pass_equals_oracle(ctx, over, vw, strong):
    g = graphgen.grid2d(91, 90, ew=(1, 50), seed=over)     # 8,190 vertices: 32 tiles
    k = 256
    g = graphgen.Graph(g.n, g.xadj, g.adjncy, np.full(g.n, vw, np.int32), g.adjwgt)
    # stripes of consecutive vertices, so that some candidates have no neighbour outside
    part = (np.arange(g.n) * over // g.n).astype(np.int32)
    ref = oracle.jetrs(g, k, part, eps=0.03) if strong else oracle.jetrw(g, k, part, eps=0.03, seed=17, it=5)
    d = [torch.as_tensor(np.asarray(a)).cuda() for a in (g.xadj, g.adjncy, g.vwgt, g.adjwgt)]
    r = ctx.rebalance_pass(*d, k, part, eps=0.03, strong=strong, seed=17, it=5)
    assert r["ncand"] == ref["ncand"] and r["nmoves"] == ref["nmoves"]
    got = r["loss"].cpu().numpy().astype(np.int64)
    cand = ref["loss"] != oracle.NONE
    assert np.array_equal(got[cand], ref["loss"][cand])
    assert np.array_equal(r["dest"].cpu().numpy(), ref["dest"])
