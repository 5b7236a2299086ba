"""JET_FLAG_NO_PDL: no kernel of a refinement, from the level's start to its
last iteration, and none of a single pass may start before the launch ahead of
it has finished.  Counted at the launches (the results do not show it)."""
import numpy as np
import pytest
import torch

import graphgen
import oracle

pytestmark = pytest.mark.gpu

jet = pytest.importorskip("paper_2304_13194_gb300")

CALLS = {
    "refine": lambda c, t, p: c.refine(*t, 16, p, seed=2),
    "lp_pass": lambda c, t, p: c.lp_pass(*t, 16, p),
    "lp_pass_noalloc": lambda c, t, p: c.lp_pass_noalloc(*t, 16, p),
    "rebalance_weak": lambda c, t, p: c.rebalance_pass(*t, 16, p, strong=False),
    "rebalance_strong": lambda c, t, p: c.rebalance_pass(*t, 16, p, strong=True),
}


@pytest.mark.parametrize("call", CALLS)
@pytest.mark.parametrize("loop", [0, jet.FLAG_HOSTLOOP, jet.FLAG_GRID_LOOP], ids=["graph", "host", "grid"])
def test_no_pdl_holds_for_every_refinement_launch(call, loop):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    g = graphgen.grid3d(20, 20, 20, vw=(1, 4), ew=(1, 10), seed=6)
    t = [torch.from_numpy(a).cuda() for a in (g.xadj, g.adjncy, g.vwgt, g.adjwgt)]
    part = torch.from_numpy(np.minimum(oracle.initial_partition(g, 16) * 3 // 2, 15).astype(np.int32)).cuda()
    counts = {}
    for flag in (0, jet.FLAG_NO_PDL):
        with jet.Context(0, flags=loop | flag, cluster_max_n=0) as c:
            before = jet.binding.early_launch_count()
            CALLS[call](c, t, part)
            counts[flag] = jet.binding.early_launch_count() - before
    assert counts[jet.FLAG_NO_PDL] == 0
    assert counts[0] > 0          # and without the flag there are some
