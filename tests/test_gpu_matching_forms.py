"""Which form matches a level: all rounds in one cluster launch, or two launches
per round, which long rows and many entries need.  The launches that may start
early tell them apart (the cluster launch is not one)."""
import numpy as np
import pytest
import torch

import graphgen
import oracle
from helpers import graph_from_triples

pytestmark = pytest.mark.gpu

jet = pytest.importorskip("paper_2304_13194_gb300")


def _hub(n, leaves):
    """A ring of n vertices, vertex 0 with `leaves` neighbours in all."""
    t = [[v, (v + 1) % n, 1 + v % 3] for v in range(n)]
    return graph_from_triples(n, t + [[0, v, 2] for v in range(2, leaves)])


FORMS = [
    ("geometric", lambda: graphgen.rgg(8000, seed=1), True),
    ("mesh_w", lambda: graphgen.grid3d(32, 32, 32, vw=(1, 4), ew=(1, 10), seed=2), True),
    ("row_128", lambda: _hub(4000, 128), True),
    ("row_129", lambda: _hub(4000, 129), False),
    ("hub_in_the_last_row", lambda: graph_from_triples(5000, [[v, v + 1, 1] for v in range(4999)] +
                                                       [[4999, 3 * v, 2] for v in range(1500)]), False),
    ("rmat_sparse", lambda: graphgen.rmat(12, 2, seed=3), False),
    ("rmat_sparse_w", lambda: graphgen.rmat(15, 1, seed=3, ew=(1, 5)), False),
    ("entries_below", lambda: graphgen.gnp(32768, 11.5 / 32768, seed=4), True),
    ("entries_above", lambda: graphgen.gnp(32768, 13.0 / 32768, seed=5), False),
]


@pytest.mark.parametrize("name,make,cluster", FORMS, ids=[f[0] for f in FORMS])
def test_form_of_the_matching(name, make, cluster):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    g = make()
    t = [torch.from_numpy(a).cuda() for a in (g.xadj, g.adjncy, g.adjwgt)]
    with jet.Context(0) as c:
        e0 = jet.binding.early_launch_count()
        mate = c.hem(*t, seed=11).cpu().numpy()
        early = jet.binding.early_launch_count() - e0
        assert np.array_equal(mate, oracle.hem(g, 11, 0, 8))
        assert early == (0 if cluster else 16)


def test_coarse_levels_with_long_rows_take_the_launches():
    """Inside a hierarchy the bound on a level's rows comes from the level before;
    the hierarchy is the oracle's."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    g, k = graphgen.rmat(16, 2, seed=6, ew=(1, 5)), 8
    with jet.Context(0) as c:
        part, cut = c.partition(g.xadj, g.adjncy, g.vwgt, g.adjwgt, k=k, seed=3)
    ref = oracle.partition(g, k, 0.03, 3)
    assert cut == ref.cut and (part.cpu().numpy() == ref.part).all()
