"""The tuner's choice for a small flexible set is no slower than the set left
alone, whose replicas the library hands to teams of warps."""
import numpy as np
import pytest

from paper_2508_15522_gb300 import synth

pytestmark = pytest.mark.gpu


def test_tuning_keeps_the_teams():
    import __graft_entry__ as ge
    ge.build()
    from paper_2508_15522_gb300 import gridff as G
    ctx = G.Context(0)
    sub = synth.rocksalt_slab(ncell=2)
    box = synth.grid_box_for(sub, 0.25, height=9.0)
    grid = G.build_grid(ctx, sub, box.origin, box.length, box.spacing)
    mol = synth.random_flexible_molecule(47, 3, 5)
    x = synth.flexible_positions(mol, sub, 64, seed=6).astype(np.float32).ravel()
    prm = G.fire_params(f_conv=0.0)

    def once(reps):
        reps.set_state(x)
        G.relax(ctx, grid, reps, 100, prm)
        return reps.get_state()[0], ctx.last_kernel_ms()

    alone, tuned = G.Replicas(ctx, [mol], [0] * 64), G.Replicas(ctx, [mol], [0] * 64)
    tuned.set_launch_config(kernel=G.KERNEL_FLEX_TERMS)      # a layout set before does not keep the heuristic out
    tuned.set_state(x)
    best, log = G.tune(ctx, grid, tuned, prm, trial_steps=50)
    assert max(t["atom_evals_per_s"] for t in log) > 0 and tuned.launch_config().kernel == best.kernel
    xa, xt, a, t = None, None, [], []
    for _ in range(7):
        xa, ms = once(alone)
        a.append(ms)
        xt, ms = once(tuned)
        t.append(ms)
    # a warp per replica takes 3 to 4 times as long as a team
    assert np.median(t[1:]) <= 1.5 * np.median(a[1:]), (t, a)
    assert np.array_equal(xa, xt)
