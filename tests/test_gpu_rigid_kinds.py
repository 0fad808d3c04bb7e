"""The sub-warp rigid kernel has a build of its own for 16-bit two-slot grids,
FP16 and BF16: its energies against the warp-per-replica kernel's, which
chooses the record kind at run time."""
import numpy as np
import pytest

from oracle import bspline as obs
from oracle import dynamics as odyn
from oracle import precision as oprec
from oracle import substrate as osub
from paper_2508_15522_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import __graft_entry__ as ge
    ge.build()
    from paper_2508_15522_gb300 import gridff as G
    ctx = G.Context(0)
    sub = synth.fcc111_slab(ncell=4, layers=3, grid_height=8.0)
    box = synth.grid_box_for(sub, 0.2, height=8.0)
    grids = {t: G.build_grid(ctx, sub, box.origin, box.length, box.spacing, channels=G.CH_P | G.CH_L,
                             keep_f64=True, storage=oprec.STORAGE[t]) for t in ("f16", "bf16")}
    return G, ctx, sub, box, grids


# atoms per lane 1 to 4, full and partial; odd replica counts leave lanes without a replica
@pytest.mark.parametrize("tier", ["f16", "bf16"])
@pytest.mark.parametrize("n, W, n_rep", [(8, 8, 5), (13, 16, 3), (24, 8, 33), (38, 16, 7), (38, 32, 2), (64, 16, 3)])
def test_energy_equals_the_quad_kernel(env, tier, n, W, n_rep):
    G, ctx, sub, box, grids = env
    g = grids[tier]
    mol = synth.rigid_molecule(n, 5)
    com, quat = synth.rigid_poses(mol, sub, n_rep, seed=n)
    pose = np.concatenate([com, quat], 1).astype(np.float32)
    E = {}
    for kernel, lanes in ((G.KERNEL_RIGID_SUBWARP, W), (G.KERNEL_RIGID_QUAD, 32)):
        reps = G.Replicas(ctx, [mol], [0] * n_rep, rigid=True)
        reps.set_launch_config(kernel=kernel, lanes_per_replica=lanes, blocks=0)
        reps.set_state(pose.ravel())
        G.relax(ctx, g, reps, 1, G.fire_params(f_conv=0.0))
        E[kernel] = reps.fire_state()["energy"].astype(np.float64)
        reps.close()
    # a 64-term stencil sum and the sum over atoms: 80 roundings of the sum of
    # absolute terms; atom positions and cell fractions (coordinates below 32 A):
    # 6e-6 A along the force in either kernel
    pos = odyn.rigid_positions(pose[:, :3].astype(np.float64), pose[:, 3:].astype(np.float64), mol.xyz).reshape(-1, 3)
    P_, L_ = osub.factor_params(np.tile(mol.R, n_rep), np.tile(mol.eps, n_rep), 1.5)
    coefs = g.download_f64("coefs")
    fa, _, _ = obs.eval_grid(np.abs(coefs), box.origin, g.spacing, pos)
    _, grad, _ = obs.eval_grid(coefs, box.origin, g.spacing, pos)
    e_abs = np.abs(P_) * fa[:, 0] + np.abs(L_) * fa[:, 1]
    f_abs = np.abs(P_[:, None] * grad[:, 0] + L_[:, None] * grad[:, 1]).sum(1)
    bound = (80 * 2.0 ** -24 * e_abs + 1.2e-5 * f_abs).reshape(n_rep, n).sum(1)
    dE = np.abs(E[G.KERNEL_RIGID_SUBWARP] - E[G.KERNEL_RIGID_QUAD])
    assert np.isfinite(dE).all() and np.all(dE <= bound)
