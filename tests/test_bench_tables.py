"""The benchmark's kernel table and refinement rate cover the levels that the
timed step refines with per-kernel launches, not those of a cluster launch."""
import os
import sys
from types import SimpleNamespace

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _stats(blocks):
    return SimpleNamespace(levels=3, cluster_blocks=blocks, ms_level=[4.0, 2.0, 1.0], ms_refine=7.5,
                           kern_bytes=[[300, 100], [200, 0], [70, 30]], kern_ms=[[0.3, 0.1], [0.5, 0.0], [0.1, 0.9]],
                           kern_launches=[[3, 1], [2, 0], [1, 2]], bytes_model=700)


@pytest.mark.parametrize("blocks,levels,byts,ms,top", [([0, 0, 16], [0, 1], 600, 6.0, "a"), ([0, 16, 0], [0, 2], 500, 5.0, "b"),
                                                       ([8, 8, 8], [0, 1, 2], 700, 7.0, "b")])
def test_tables_leave_out_the_levels_of_a_cluster_launch(blocks, levels, byts, ms, top):
    sys.path.insert(0, ROOT)
    import bench
    st, prof = _stats(blocks), _stats([0, 0, 0])
    assert bench.kernel_levels(st) == levels
    assert bench.refine_rate(st) == pytest.approx(byts / (ms / 1e3) / 1e9)
    table, name = bench.kernel_table(prof, ["a", "b"], 1.0, bench.kernel_levels(st))
    assert name == top
    assert sum(r["bytes"] for r in table.values()) == byts
    assert sum(r["launches"] for r in table.values()) == sum(sum(prof.kern_launches[i]) for i in levels)
