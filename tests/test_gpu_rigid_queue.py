"""Rigid relaxations that may stop early take their tasks from a queue, in parts
of equal iteration ranges where whole tasks would leave warps idle: bit for bit
the result of whole tasks in one launch per part, whatever converges on the way
and however the launch is capped."""
import numpy as np
import pytest

from paper_2508_15522_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import __graft_entry__ as ge
    ge.build()
    from paper_2508_15522_gb300 import gridff as G
    ctx = G.Context(0)
    sub = synth.rocksalt_slab(ncell=2)
    box = synth.grid_box_for(sub, 0.25, height=9.0)
    return G, ctx, sub, G.build_grid(ctx, sub, box.origin, box.length, box.spacing)


# blocks: 1 to 3 blocks of 4 warps share 57 or 129 tasks; n_rep odd: the last task
# is partly empty.  nsteps 200 and 333: parts of unequal length
@pytest.mark.parametrize("n_rep, blocks, nsteps, f_conv", [(113, 1, 200, 1e-3), (257, 3, 333, 1e-3), (257, 2, 200, 0.5),
                                                           (113, 3, 64, 0.05)])
def test_parts_equal_whole_tasks(env, n_rep, blocks, nsteps, f_conv):
    G, ctx, sub, grid = env
    mol = synth.c24h8o6_core()
    com, quat = synth.rigid_poses(mol, sub, n_rep, seed=n_rep)
    pose = np.concatenate([com, quat], 1).astype(np.float32).ravel()
    out = []
    for cap in (blocks, 0):          # capped: more tasks than warps, in parts; uncapped: a warp for every task
        reps = G.Replicas(ctx, [mol], [0] * n_rep, rigid=True)
        cfg = reps.launch_config()
        cfg.lanes_per_replica, cfg.blocks = 16, cap
        reps.set_launch_config(cfg)
        reps.set_state(pose)
        _, res = G.relax(ctx, grid, reps, nsteps, G.fire_params(f_conv=f_conv))
        fs = reps.fire_state()
        out.append((reps.get_state(), reps.last_eval(), fs, res.atom_evals, res.n_converged, res.max_steps))
        assert res.atom_evals == int(fs["steps"].sum()) * mol.n
        assert res.n_converged == int(((fs["status"] & G.REP_CONVERGED) != 0).sum())
    a, b = out
    assert np.array_equal(a[0][0], b[0][0]) and np.array_equal(a[0][1], b[0][1])
    assert np.array_equal(a[1][0], b[1][0]) and np.array_equal(a[1][1], b[1][1])
    assert all(np.array_equal(a[2][k], b[2][k]) for k in a[2]) and a[3:] == b[3:]
    if f_conv == 0.5:
        assert 0 < a[4] < n_rep      # some replicas stop in an early part


def test_parts_stop_on_abort(env):
    G, ctx, sub, grid = env
    mol = synth.c24h8o6_core()
    com, quat = synth.rigid_poses(mol, sub, 113, seed=3)
    reps = G.Replicas(ctx, [mol], [0] * 113, rigid=True)
    reps.set_launch_config(lanes_per_replica=16, blocks=1)
    reps.set_state(np.concatenate([com, quat], 1).astype(np.float32).ravel())
    ctx.set_abort(True)
    try:
        st, res = G.relax(ctx, grid, reps, 200, G.fire_params(f_conv=1e-3), check=False)
    finally:
        ctx.set_abort(False)
    fs = reps.fire_state()
    assert st == G.EABORTED and res.atom_evals == 0 and (fs["steps"] == 0).all()
    assert ((fs["status"] & G.REP_ABORTED) != 0).all()
    st, res = G.relax(ctx, grid, reps, 50, G.fire_params(f_conv=1e-3))
    assert st == G.OK and res.atom_evals == 50 * 113 * mol.n
