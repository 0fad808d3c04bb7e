"""Flexible batches a little above one round of warps: the first replicas of the
cost order go to the warp kernel, the others to teams, within one call.  With
molecules whose teams do not all fit the chip at once, every replica is still
served exactly once, by relaxation, its captured graph, Langevin and NVE
dynamics; and the two kernels share one clock budget."""
import numpy as np
import pytest

from paper_2508_15522_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import __graft_entry__ as ge
    ge.build()
    from paper_2508_15522_gb300 import gridff
    import torch
    return gridff, gridff.Context(0), 32 * torch.cuda.get_device_properties(0).multi_processor_count


def dense_molecule(n=120):
    """All angles and torsions of the bond graph: a team of 4 warps needs more
    than 57 kB of shared memory, so three fit an SM (456 on 152)."""
    m = synth.random_flexible_molecule(n, 3, 7)
    m = synth._finish(m.elements, m.xyz, m.q, m.bonds)
    assert len(m.bonds) + 3 * len(m.angles) + 4 * len(m.torsions) >= 1500
    return m


@pytest.fixture(scope="module")
def batch(env):
    """With the grid: its stencils are part of a team's shared memory."""
    G, ctx, W = env
    sub = synth.rocksalt_slab(ncell=2)
    box = synth.grid_box_for(sub, 0.3, height=14.0)
    grid = G.build_grid(ctx, sub, box.origin, box.length, box.spacing)
    mol = dense_molecule()
    n_rep = W + W // 8 - 100           # 508 replicas past one round of 4864
    g = np.random.default_rng(11)
    low = mol.xyz[:, 2].min() - sub.z_top - 3.0
    x = (mol.xyz[None] - [0.0, 0.0, low] + g.normal(0.0, 0.02, (n_rep, mol.n, 3))).astype(np.float32)
    return mol, n_rep, x.ravel(), grid


# Positions of the two layouts differ by the order of FP32 sums: 1e-5 A after
# three steps, the bound of the small-batch test of the same split.
@pytest.mark.parametrize("call", ["relax", "graph", "langevin", "run"])
def test_every_replica_is_served_once(env, batch, call):
    G, ctx, _ = env
    mol, n_rep, x, grid = batch
    out = []
    for split in (True, False):
        reps = G.Replicas(ctx, [mol], [0] * n_rep)
        if not split:
            reps.set_launch_config(kernel=G.KERNEL_FLEX_TERMS)
        reps.set_state(x)
        trace = None
        if call == "relax":
            _, res = G.relax(ctx, grid, reps, 3, G.fire_params(f_conv=0.0))
        elif call == "graph":
            graph = G.RelaxGraph(ctx, grid, reps, 3, G.fire_params(f_conv=0.0))
            _, res = graph.launch()
            graph.close()
        elif call == "langevin":
            G.langevin(ctx, grid, reps, 3, 0.5, 300.0, 0.01, seed=4)
        else:
            _, trace = G.run(ctx, grid, reps, 3, 0.5, record_every=1)
        fs = reps.fire_state()
        if call in ("relax", "graph"):
            assert (fs["steps"] == 3).all(), int((fs["steps"] != 3).sum())
            assert res.atom_evals == 3 * mol.n * n_rep
        out.append((reps.get_state()[0], fs["energy"], trace))
        reps.close()
    (x1, e1, t1), (x0, e0, t0) = out
    assert np.abs(x1 - x0).max() <= 1e-5
    assert (np.abs(e1 - e0) <= 1e-5 * np.maximum(mol.n, np.abs(e0))).all()
    if t0 is not None:
        assert (np.abs(t1 - t0) <= 1e-5 * np.maximum(mol.n, np.abs(t0))).all()


@pytest.mark.parametrize("call", ["relax", "langevin", "run"])
def test_one_clock_budget(env, batch, call):
    """The budget counts from the call's first kernel: the second one, which
    starts when the first has used it up, stops at once.  200 ms against the
    400 ms of two budgets; 100 ms allow for the 32 steps between looks at the
    clock (3 ms) and the launches."""
    G, ctx, _ = env
    mol, n_rep, x, grid = batch
    reps = G.Replicas(ctx, [mol], [0] * n_rep)
    for budget in (0.01, 0.2):         # the first call warms up
        reps.set_state(x)
        if call == "relax":
            st, _ = G.relax(ctx, grid, reps, 10**8, G.fire_params(f_conv=0.0, clock_budget_s=budget),
                            check=False)
        elif call == "langevin":
            st = G.langevin(ctx, grid, reps, 10**8, 0.1, 10.0, 0.01, seed=4, clock_budget_s=budget,
                            check=False)
        else:
            st, _ = G.run(ctx, grid, reps, 10**8, 0.1, clock_budget_s=budget, check=False)
        assert st == G.ESTEPLIMIT
    assert 200.0 <= ctx.last_kernel_ms() <= 300.0
    assert ((reps.fire_state()["status"] & G.REP_STEPLIMIT) != 0).all()


@pytest.mark.parametrize("sizes, rounds, split", [((22,), 1, True), ((44, 47), 2, True), ((113, 120), 1, True),
                                                  ((113, 120), 2, False), ((10, 60, 120), 1, False), ((30, 47), 1, False)])
def test_which_last_rounds_go_to_teams(env, batch, sizes, rounds, split):
    """Only those of even batches, where a team is faster than the queue: seen by the
    bits, which differ between the layouts in the order of FP32 sums."""
    G, ctx, W = env
    grid = batch[3]
    sub = synth.rocksalt_slab(ncell=2)
    mols = [synth.random_flexible_molecule(n, 3, n) for n in sizes]
    n_rep = rounds * W + 37
    tof = np.arange(n_rep) % len(mols)
    pos = [synth.flexible_positions(m, sub, 8, seed=3).astype(np.float32).reshape(8, -1) for m in mols]
    x = np.concatenate([pos[k][i % 8] for i, k in enumerate(tof)])
    out = []
    for default in (True, False):
        reps = G.Replicas(ctx, mols, tof)
        if not default:
            reps.set_launch_config(kernel=G.KERNEL_FLEX_TERMS)
        reps.set_state(x)
        G.relax(ctx, grid, reps, 4, G.fire_params(f_conv=0.0))
        out.append(reps.last_eval()[1])
        off = reps.atom_offset
        reps.close()
    d = np.abs(out[0] - out[1]).max(1)
    differ = sum(d[off[r]:off[r + 1]].any() for r in range(n_rep))
    assert differ <= 37 and (differ > 30 if split else differ == 0)
