"""Dynamics take every layout that a relaxation takes: a warp of md_flex keeps
velocities too, so a stencil staging that just fits a relaxation has to be cut
down, which changes no result."""
import numpy as np
import pytest

from paper_2508_15522_gb300 import synth

pytestmark = pytest.mark.gpu


def test_the_largest_staging_of_a_relaxation():
    import __graft_entry__ as ge
    ge.build()
    from paper_2508_15522_gb300 import gridff as G
    ctx = G.Context(0)
    sub = synth.rocksalt_slab(ncell=2)
    box = synth.grid_box_for(sub, 0.25, height=9.0)
    grid = G.build_grid(ctx, sub, box.origin, box.length, box.spacing)
    mol = synth.random_flexible_molecule(100, 3, 5)
    x = synth.flexible_positions(mol, sub, 3, seed=6).astype(np.float32).ravel()
    v = (1e-3 * np.random.default_rng(1).standard_normal(x.size)).astype(np.float32)
    out = []
    for slots in (88, 0):
        reps = G.Replicas(ctx, [mol], [0] * 3)
        reps.set_launch_config(kernel=G.KERNEL_FLEX_TERMS, warps_per_block=8, cache_slots=slots, cache_global=0)
        reps.set_state(x, v)
        G.relax(ctx, grid, reps, 1, G.fire_params(f_conv=0.0))
        reps.set_state(x, v)
        _, trace = G.run(ctx, grid, reps, 5, 0.5, record_every=5)
        xr = reps.get_state()[0]
        reps.set_state(x, v)
        G.langevin(ctx, grid, reps, 5, 0.5, 300.0, 0.01, seed=3)
        out.append((trace, xr, reps.get_state()[0]))
    for a, b in zip(*out):           # staged stencils hold the values that a gather gives
        assert np.abs(a - b).max() <= 1e-6 * max(1.0, np.abs(b).max())
