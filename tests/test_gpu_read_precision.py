"""Precision of the results that are read (evaluations and constant-energy
dynamics), in both splits of a replica over lanes (a warp; a team of warps):
no worse than the per-atom pass with its divisions, FP64 sums of the energies,
and the velocity update with the mass as divisor."""
import numpy as np
import pytest

from oracle import intra as ointra
from paper_2508_15522_gb300 import synth

pytestmark = pytest.mark.gpu
f32 = np.float32
KE = f32(14.399645)
ACC = f32(9.648533e-3)

# replicas that go to teams, and to a warp each (more than 8 per SM)
SPLITS = (200, 1300)


@pytest.fixture(scope="module")
def env():
    import __graft_entry__ as ge
    ge.build()
    from paper_2508_15522_gb300 import gridff
    return gridff, gridff.Context(0)


def molecule(n, q=None, mass=None, **terms):
    """n atoms without nonbonded wells; charges and bonded terms as given (FP32 values)."""
    m = synth.Molecule(["C"] * n, np.zeros((n, 3)), np.zeros(n) if q is None else q, np.ones(n), np.zeros(n),
                       np.full(n, 12.0) if mass is None else mass)
    for k, v in terms.items():
        setattr(m, k, v)
    return m


@pytest.mark.parametrize("n_rep", SPLITS)
def test_pair_energies_are_summed_in_fp64(env, n_rep):
    """128 like charges: all pair energies of one sign, so that long FP32 sums show.
    Relative spread of the energy's error over replicas: 4.8e-9 for FP32 sums over 32
    partners at most, 1.85e-8 for sums over up to 128 (numpy, terms of 1.2e-7 rms
    error); 9e-9 between them."""
    G, ctx = env
    n = 128
    g = np.random.default_rng(3)
    q = (0.3 + 0.2 * g.random(n)).astype(f32)
    x = (12 * g.random((n_rep, n, 3))).astype(f32)
    reps = G.Replicas(ctx, [molecule(n, q.astype(float))], [0] * n_rep)
    reps.set_state(x.ravel())
    E = G.eval(ctx, None, reps, flags=G.NO_GRID)[0][:200]
    X = x[:200].astype(np.float64)
    r = np.sqrt(((X[:, :, None] - X[:, None]) ** 2).sum(-1))
    pair = np.triu(np.ones((n, n), bool), 1)
    qq = (KE * q).astype(f32).astype(np.float64)[:, None] * q.astype(np.float64)[None]
    ref = np.array([(qq[pair] / rr[pair]).sum() for rr in r])
    rel = E / ref - 1
    assert np.std(rel) <= 9e-9 and abs(rel.mean()) <= 1e-7


@pytest.mark.parametrize("n_rep", SPLITS)
@pytest.mark.parametrize("term", ["angle", "torsion"])
def test_bonded_forces_as_the_per_atom_pass(env, term, n_rep):
    """One angle (torsion) per group of atoms, so that no sums blur it: the median relative
    error of an atom's force is at most 1.1 times that of the per-atom layout, whose
    reciprocals are divisions (the same number of roundings; 1.1 for their order)."""
    G, ctx = env
    per, k = (3, 42) if term == "angle" else (4, 32)
    n = per * k
    idx = np.arange(n, dtype=np.int32).reshape(k, per)
    g = np.random.default_rng(7)
    if term == "angle":
        m = molecule(n, angles=idx, angle_k=np.full(k, 3.0), angle_cos0=np.full(k, -0.25))
    else:
        m = molecule(n, torsions=idx, torsion_V=np.full(k, 0.5), torsion_n=np.full(k, 3, np.int32),
                     torsion_cos_nphi0=np.full(k, -1.0))
    # bond vectors of 1.1 to 1.6 A in random directions, groups 20 A apart in z
    step = g.standard_normal((n_rep, k, per, 3))
    step *= (1.1 + 0.5 * g.random((n_rep, k, per, 1))) / np.linalg.norm(step, axis=-1, keepdims=True)
    x = np.cumsum(step, 2)
    x[..., 2] += 20.0 * np.arange(k)[None, :, None]
    x = x.reshape(n_rep, n, 3).astype(f32)
    ref = ointra.energy_forces(x[:200].astype(np.float64), m)[1]
    err = {}
    for name in ("eval", "per atom"):
        reps = G.Replicas(ctx, [m], [0] * n_rep)
        if name == "per atom":
            reps.set_launch_config(kernel=G.KERNEL_FLEX_QUAD, warps_per_block=4, queue=0)
        reps.set_state(x.ravel())
        if name == "eval":
            F = G.eval(ctx, None, reps, flags=G.NO_GRID)[1]
        else:
            G.relax(ctx, None, reps, 1, G.fire_params(f_conv=0.0), flags=G.NO_GRID)
            F = reps.last_eval()[1]
        F = F.reshape(n_rep, n, 3)[:200].astype(np.float64)
        err[name] = np.median(np.linalg.norm(F - ref, axis=-1) / np.linalg.norm(ref, axis=-1))
    print(term, n_rep, err)
    assert err["eval"] <= 1.1 * err["per atom"]


@pytest.mark.parametrize("n_rep", SPLITS)
def test_bonded_energies_are_summed_in_fp64(env, n_rep):
    """600 bonds on a line whose energies are FP32 numbers exactly (odd multiples of 2^-22
    with 22 bits): their FP64 sum is exact, an FP32 sum of a few is not."""
    G, ctx = env
    n, k = 128, 600
    g = np.random.default_rng(5)
    pairs = np.array([(i, j) for i in range(n) for j in range(i + 1, n)], np.int32)
    bonds = pairs[np.sort(g.choice(len(pairs), k, replace=False))]
    dr = (2 * g.integers(512, 1024, k) + 1) / 2048.0
    r = (bonds[:, 1] - bonds[:, 0]).astype(float)
    m = molecule(n, bonds=bonds, bond_k=np.ones(k), bond_r0=r - dr)
    assert ((r - dr).astype(f32).astype(float) == r - dr).all() and ((dr ** 2).astype(f32).astype(float) == dr ** 2).all()
    x = np.zeros((n_rep, n, 3), f32)
    x[:, :, 0] = np.arange(n)
    reps = G.Replicas(ctx, [m], [0] * n_rep)
    reps.set_state(x.ravel())
    E = G.eval(ctx, None, reps, flags=G.NO_GRID)[0]
    assert (E == (dr ** 2).sum()).all()


@pytest.mark.parametrize("layout", ["team", "warp"])
def test_velocity_update_divides_by_the_mass(env, layout):
    """A bond that pulls the atom at x = 0 with exactly 1 eV/A: after one step of 1 fs its
    coordinate is dt/2 ACC / m rounded once, as FP32 arithmetic gives it."""
    G, ctx = env
    masses = (1.0 + 200.0 * np.random.default_rng(9).random(100)).astype(f32)
    mols = [molecule(2, mass=np.array([m, m], float), bonds=np.array([[0, 1]], np.int32), bond_k=np.ones(1),
                     bond_r0=np.full(1, 0.5)) for m in masses]
    reps = G.Replicas(ctx, mols, np.arange(100))
    if layout == "warp":
        reps.set_launch_config(kernel=G.KERNEL_FLEX_TERMS)
    x = np.zeros((100, 2, 3), f32)
    x[:, 1, 0] = 1.0
    reps.set_state(x.ravel())
    G.run(ctx, None, reps, 1, 1.0, flags=G.NO_GRID)
    got = reps.get_state()[0].reshape(100, 2, 3)[:, 0, 0]
    assert np.array_equal(got, f32(0.5) * f32(1.0) * ACC / masses)
