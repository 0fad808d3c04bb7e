"""The bounded wait of the rigid queue's hand-off bounds one part, not all parts
before it, and a captured relaxation reports a wait that ran out."""
import numpy as np
import pytest

from paper_2508_15522_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import __graft_entry__ as ge
    ge.build()
    from paper_2508_15522_gb300 import gridff as G
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ctx = G.Context(0)
    sub = synth.rocksalt_slab(ncell=2)
    box = synth.grid_box_for(sub, 0.25, height=9.0)
    return G, ctx, sub, G.build_grid(ctx, sub, box.origin, box.length, box.spacing), sms


def test_a_straggler_may_take_longer_than_the_wait(env):
    """One replica of 16 lanes iterates 1.2 million times (over 2 s; FP32 rounding keeps
    its force above 1e-12) while all others, above the grid and free of force, have
    converged: the idle warps hold its later parts, each waiting for those before it.
    The last of them is reached after more than the wait's one second."""
    G, ctx, sub, grid, sms = env
    mol = synth.c24h8o6_core()
    blocks, nsteps = sms, 1_200_000
    n_rep = 2 * (4 * blocks + 40)       # a few more tasks of two replicas than warps
    com, quat = synth.rigid_poses(mol, sub, n_rep, seed=2)
    pose = np.concatenate([com, quat], 1).astype(np.float32)
    pose[1:, 2] += 100.0
    reps = G.Replicas(ctx, [mol], [0] * n_rep, rigid=True)
    cfg = reps.launch_config()
    cfg.lanes_per_replica, cfg.blocks, cfg.queue = 16, blocks, 1
    reps.set_launch_config(cfg)
    reps.set_state(pose.ravel())
    st, res = G.relax(ctx, grid, reps, nsteps, G.fire_params(f_conv=1e-12), check=False)
    steps = reps.fire_state()["steps"]
    assert st == G.OK and steps[0] == nsteps and (steps[1:] == 1).all()
    assert ctx.last_kernel_ms() > 1200.0          # else the case does not reach the wait
    assert res.n_converged == n_rep - 1


def test_a_captured_relaxation_reports_the_wait(env):
    """With the hook that publishes no hand-off, the second parts give up (6 tasks cut
    into ranges for 4 warps); the replay says so as the direct call does."""
    G, ctx, sub, grid, sms = env
    mol = synth.c24h8o6_core()
    com, quat = synth.rigid_poses(mol, sub, 11, seed=2)
    reps = G.Replicas(ctx, [mol], [0] * 11, rigid=True)
    cfg = reps.launch_config()
    cfg.lanes_per_replica, cfg.blocks, cfg.queue = 16, 1, 2
    reps.set_launch_config(cfg)
    reps.set_state(np.concatenate([com, quat], 1).astype(np.float32).ravel())
    graph = G.RelaxGraph(ctx, grid, reps, 100, G.fire_params(f_conv=0.0), flags=G.TEST_NO_HANDOFF)
    st, _ = graph.launch(check=False)
    assert st == G.ETIMEOUT
    graph.close()
    st, res = G.relax(ctx, grid, reps, 100, G.fire_params(f_conv=0.0), check=False)
    assert st == G.OK and res.atom_evals == 11 * mol.n * 100
