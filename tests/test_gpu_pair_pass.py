"""Force pass of the flexible kernels at the molecule sizes where its blocks
and rings change, in every split of a replica over warps (one warp; teams of
2, 4 and 8), through relaxation, evaluation, NVE and Langevin dynamics.

Forces and energies of one evaluation against the oracle's FP64 force field,
held to the parity gates of every flexible kernel (1e-4 eV/A, 1e-5 eV per
atom); positions after four steps of dynamics to 1e-5 A (four half-steps of
FP32 rounding of 10 A coordinates, 1e-6 A each, and the force gate's
1e-4 eV/A x dt^2 / m = 1e-6 A on a hydrogen)."""
import numpy as np
import pytest

from oracle import dynamics as odyn
from oracle import intra as ointra
from paper_2508_15522_gb300 import synth

pytestmark = pytest.mark.gpu

# half rings of even and odd size; a full block; a second block of 1, 2, 3, 8,
# 9, 16 and 17 atoms; three and four blocks; the largest molecule
SIZES = (4, 5, 9, 16, 17, 22, 31, 32, 33, 34, 35, 40, 41, 48, 49, 64, 65, 81, 97, 128)


@pytest.fixture(scope="module")
def env():
    import __graft_entry__ as ge
    ge.build()
    from paper_2508_15522_gb300 import gridff
    return gridff, gridff.Context(0)


def as32(m):
    """The molecule with the FP32 parameters that the library is given."""
    return synth.Molecule(**{**vars(m), **{a: np.asarray(getattr(m, a), np.float32).astype(np.float64) for a in (
        "q", "R", "eps", "mass", "bond_k", "bond_r0", "angle_k", "angle_cos0", "torsion_V", "torsion_cos_nphi0")}})


@pytest.fixture(scope="module")
def cases():
    out = {}
    g = np.random.default_rng(5)
    for n in SIZES:
        m = synth.random_flexible_molecule(n, 3, 900 + n)
        x = (m.xyz + g.normal(0.0, 0.05, m.xyz.shape)).astype(np.float32)
        out[n] = (m, as32(m), x, *ointra.energy_forces(x[None].astype(np.float64), as32(m)))
    return out


# largest molecule, replicas: teams of 8; 4; 4; 2; one warp each
@pytest.mark.parametrize("largest, replicas", [(128, 20), (65, 400), (32, 700), (32, 1300), (128, 1300)])
def test_forces_at_the_block_edges(env, cases, largest, replicas):
    G, ctx = env
    sizes = [n for n in SIZES if n <= largest]
    mols = [cases[n][0] for n in sizes]
    tof = np.tile(np.arange(len(mols)), -(-replicas // len(mols))).astype(np.int32)
    reps = G.Replicas(ctx, mols, tof)
    x0 = np.concatenate([cases[sizes[t]][2] for t in tof])
    off = reps.atom_offset

    def check(E, F):
        for k, n in enumerate(sizes):
            Er, Fr = cases[n][3][0], cases[n][4][0]
            for r in (k, len(tof) - len(mols) + k):
                dF = np.abs(F[off[r]:off[r + 1]] - Fr).max()
                assert dF <= 1e-4 * max(1.0, np.abs(Fr).max()), (n, dF)
                assert abs(E[r] - Er) <= 1e-5 * max(n, abs(Er)), (n, E[r], Er)

    reps.set_state(x0.ravel())
    G.relax(ctx, None, reps, 1, G.fire_params(f_conv=0.0), flags=G.NO_GRID)
    check(reps.fire_state()["energy"], reps.last_eval()[1])
    reps.set_state(x0.ravel())
    E, F, _, _ = G.eval(ctx, None, reps, flags=G.NO_GRID)
    check(E, F)


@pytest.mark.parametrize("layout", ["team", "warp"])
@pytest.mark.parametrize("n", [5, 17, 33])
def test_dynamics_of_both_layouts(env, cases, layout, n):
    G, ctx = env
    mol, m32, x0, _, _ = cases[n]
    reps = G.Replicas(ctx, [mol], [0] * 3)
    if layout == "warp":
        reps.set_launch_config(kernel=G.KERNEL_FLEX_TERMS)
    g = np.random.default_rng(n)
    v0 = (g.standard_normal((3, n, 3)) * np.sqrt(0.025852 * 9.648533e-3 / mol.mass)[None, :, None]).astype(np.float32)
    X, V = np.repeat(x0[None], 3, 0).astype(np.float64), v0.astype(np.float64)

    def force(x):
        return (*ointra.energy_forces(x, m32), None)

    reps.set_state(X.astype(np.float32).ravel(), v0.ravel())
    _, trace = G.run(ctx, None, reps, 4, 1.0, record_every=2, flags=G.NO_GRID)
    xr, _, tr = odyn.nve_flexible(X, V, m32.mass, force, 4, 1.0, record_every=2)
    assert np.abs(reps.get_state()[0].reshape(3, n, 3) - xr).max() <= 1e-5
    assert trace.shape == tr.shape and np.abs(trace - tr).max() <= 1e-5 * n
    reps.set_state(X.astype(np.float32).ravel(), v0.ravel())
    G.langevin(ctx, None, reps, 4, 1.0, 300.0, 0.01, seed=9, step0=2, flags=G.NO_GRID)
    xr, _, er = odyn.langevin_baoab(X, V, m32.mass, force, 4, 1.0, 300.0, 0.01,
                                    lambda s: odyn.langevin_noise(9, range(3), s + 2, 3 * n))
    assert np.abs(reps.get_state()[0].reshape(3, n, 3) - xr).max() <= 1e-5
    assert np.abs(reps.fire_state()["energy"] - er).max() <= 1e-5 * n


def test_a_small_last_round_goes_to_teams(env, cases):
    """Slightly more replicas than one round of warps: both kernels of the
    split give the single-warp layout's result, every replica once."""
    G, ctx = env
    mol, _, x0, _, _ = cases[9]
    import torch
    n_rep = 32 * torch.cuda.get_device_properties(0).multi_processor_count + 5
    x = np.tile(x0.ravel(), n_rep).reshape(n_rep, -1) + 1e-3 * np.arange(n_rep)[:, None] / n_rep
    out = []
    for split in (True, False):
        reps = G.Replicas(ctx, [mol], [0] * n_rep)
        if not split:
            reps.set_launch_config(kernel=G.KERNEL_FLEX_TERMS)
        reps.set_state(x.astype(np.float32).ravel())
        _, res = G.relax(ctx, None, reps, 3, G.fire_params(f_conv=0.0), flags=G.NO_GRID)
        assert res.atom_evals == 3 * 9 * n_rep and (reps.fire_state()["steps"] == 3).all()
        out.append(reps.get_state()[0])
    assert np.abs(out[0] - out[1]).max() <= 1e-5
