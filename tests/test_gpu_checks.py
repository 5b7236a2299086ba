"""Input checks and start values on arrays at every alignment: weight sums and
part range over flat arrays whose length and address are no multiple of a
16-byte load, and the level start's copies of such a part vector."""
import numpy as np
import pytest
import torch

import graphgen
import oracle

pytestmark = pytest.mark.gpu

jet = pytest.importorskip("paper_2304_13194_gb300")


def _shifted(a, off):
    """Device copy of `a` that starts `off` entries past an aligned address."""
    buf = torch.zeros(len(a) + off, dtype=torch.from_numpy(a[:0]).dtype, device="cuda")
    buf[off:] = torch.from_numpy(a).cuda()
    return buf[off:]


@pytest.mark.parametrize("n", [1, 3, 4, 31, 1025, 4099])
@pytest.mark.parametrize("off", [0, 1, 3])
def test_checks_and_cut_at_every_alignment(n, off):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    g = graphgen.rgg(n, seed=n, vw=(1, 4), ew=(1, 10))
    k = 5
    part = np.random.default_rng(n).integers(0, k, n).astype(np.int32)
    x, a, vw, ew, p = (torch.from_numpy(g.xadj).cuda(), _shifted(g.adjncy, off), _shifted(g.vwgt, off),
                       _shifted(g.adjwgt, off), _shifted(part, off))
    with jet.Context(0) as c:
        for _ in range(2):                      # the checks' state is clear again after each call
            cut, pw = c.cut(x, a, vw, ew, k, p)
            assert cut == oracle.cut(g, part) and (pw.cpu().numpy() == oracle.part_weights(g, part, k)).all()
        for bad in (-1, k):                     # the last vertex's part out of range
            q = p.clone()
            q[n - 1] = bad
            with pytest.raises(jet.JetError) as ei:
                c.cut(x, a, vw, ew, k, q)
            assert ei.value.status == -1
        if n > 31:                              # the sums' limit, reached by the last entries alone
            w = ew.clone()
            w[-2:] = 2 ** 30
            with pytest.raises(jet.JetError) as ei:
                c.cut(x, a, vw, w, k, p)
            assert ei.value.status == -6
        cut, _ = c.cut(x, a, vw, ew, k, p)      # and the context still works
        assert cut == oracle.cut(g, part)
        got = c.lp_pass(x, a, vw, ew, k, p)
        ref = oracle.jetlp(g, k, part)
        assert (got["Pd"].cpu().numpy() == ref["Pd"]).all() and (got["inM"].cpu().numpy() == ref["inM"]).all()
