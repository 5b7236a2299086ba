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
