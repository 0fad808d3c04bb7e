"""Grids of fewer work items than the chip has warps: the items are spread over
all SMs, so a node costs about what it costs in a larger grid."""
import time

import numpy as np
import pytest

from paper_2508_15522_gb300 import synth

pytestmark = pytest.mark.gpu


def test_a_node_of_a_small_grid_costs_no_more():
    """Cutoff beyond the radial table (the functions called directly), 75 x 75 x 27 nodes
    against 8 times as many, which fill the chip many times over: the time per node
    is at most 2.5 times the large grid's (3 to 5 where a part of the SMs has no work)."""
    import __graft_entry__ as ge
    ge.build()
    from paper_2508_15522_gb300 import gridff as G
    ctx = G.Context(0)
    sub = synth.rocksalt_slab(ncell=4)
    per_node = []
    for spacing in (0.3, 0.15):
        box = synth.grid_box_for(sub, spacing, height=8.0)
        n = np.prod([np.ceil(length / spacing - 1e-9) for length in box.length])
        t = []
        for _ in range(5):
            t0 = time.perf_counter()
            grid = G.build_grid(ctx, sub, box.origin, box.length, box.spacing, rcut=25.0)
            t.append(time.perf_counter() - t0)
            grid.close()
        per_node.append(np.median(t[1:]) / n)
    ctx.close()
    assert per_node[0] <= 2.5 * per_node[1], per_node
