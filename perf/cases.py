"""What a user of this library has it do, as cases that can be timed and compared.

The work is the method's: building a substrate grid, evaluating it (alone or
with the molecule's own force field), relaxing and propagating many replicas of
rigid or flexible molecules over it, and training the network that proposes
their starting poses.  Sizes are those of the benchmark, the tests and the
examples of this repository, from one interactive handful of replicas to the
full batches.

A pass sets the start (device to device, as a sampling loop does), runs one
library call and copies the whole result into the caller's device arrays.
Trajectories are cut short enough (steps below) that FP32 rounding has not yet
grown into different paths: the outputs can be compared value by value.
Energies come out of the library as FP64 sums of FP32 terms; they are handed on
in FP32, the precision that they carry.

`exact` restates every case in 64 bits with plain torch, from the same inputs:
direct Morse sums, the closed two-dimensional Fourier sum of a neutral-layer
slab for the Coulomb channel, the exact spline fit, the force field by
differentiation of its energy, and the integrators by their definitions.
"""
from __future__ import annotations

import ctypes
import functools
import math

import numpy as np
import torch

from paper_2508_15522_gb300 import gridff as G
from paper_2508_15522_gb300 import synth

ACC = 9.648533e-3        # A/fs^2 per eV/(A amu)
KE = 14.399645           # eV A / e^2
KB = 8.617333262e-5      # eV/K
ALPHA, RCUT = 1.5, 17.0  # Morse exponent (1/A) and cutoff (A) of the substrate sums
NET = (80, 256, 256, 256, 19)
STORE = {"f32": G.STORE_F32, "f16": G.STORE_F16, "bf16": G.STORE_BF16}
DEV = "cuda"


def listed():
    return [
        # an interactive session: a handful of small molecules dropped on a surface
        dict(name="relax rigid 64 x 10", kind="relax_rigid", field="nacl", storage="f32", replicas=64, atoms=10, steps=200),
        # the headline: 4096 poses of the 38-atom core on NaCl
        dict(name="relax rigid 4096 x 38", kind="relax_rigid", field="nacl", storage="f32", replicas=4096, atoms=38, steps=200),
        # the precision-tier batch: two-channel FP16 grid over a metal surface
        dict(name="relax rigid 65536 x 24 f16", kind="relax_rigid", field="fcc", storage="f16", replicas=65536, atoms=24, steps=50),
        # energy-conserving dynamics of adsorbed molecules, an odd batch
        dict(name="run rigid 1001 x 38", kind="run_rigid", field="nacl", storage="f32", replicas=1001, atoms=38, steps=200),
        # a few conformers of one flexible molecule (the hopping molecule's size)
        dict(name="relax flexible 64 x 22", kind="relax_flex", field="hard", storage="f32", replicas=64, atoms=22, steps=16),
        # the uneven batch: 10 to 120 atoms in one launch
        dict(name="relax flexible 16384 uneven", kind="relax_flex", field="nacl", storage="f32", replicas=16384, atoms=0, steps=16),
        # a short stretch of constant-energy dynamics between two frames
        dict(name="run flexible 1024 x 47", kind="run_flex", field="hard", storage="f32", replicas=1024, atoms=47, steps=10),
        # the thermalisation of minima hopping, the paper's replica count
        dict(name="langevin 5000 x 22", kind="langevin", field="hard", storage="f32", replicas=5000, atoms=22, steps=20),
        # single-point energies and forces of a batch, for an integrator outside
        dict(name="eval flexible 4097 uneven", kind="eval", field="nacl", storage="f32", replicas=4097, atoms=0),
        # the grid alone at independent points (the interpolation benchmark's count)
        dict(name="points 2490368", kind="points", field="nacl", storage="f32", points=2490368, binned=False),
        # training the pose-proposal network: batches of 256 targets, 8 proposals each
        dict(name="train 256 x 8", kind="train", targets=256, proposals=8, steps=20),
        # the grid of a new substrate at the benchmark's spacing
        dict(name="build 113 x 113 x 208", kind="build", cells=8, layers=3, spacing=0.1),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["relax_rigid", "run_rigid", "relax_flex", "run_flex", "langevin", "eval", "points", "train", "build"])
    if kind == "points":
        return dict(kind=kind, field=rng.choice(["nacl", "fcc"]), storage=rng.choice(["f32", "f16"]),
                    points=log_int(1000, 2490368), binned=rng.random() < 0.5)
    if kind == "train":
        return dict(kind=kind, targets=log_int(16, 256), proposals=rng.randint(1, 8), steps=rng.randint(2, 20))
    if kind == "build":
        return dict(kind=kind, cells=rng.choice([2, 4, 6, 8]), layers=rng.randint(1, 3), spacing=rng.uniform(0.12, 0.4))
    if kind in ("relax_rigid", "run_rigid"):
        atoms = log_int(5, 120)
        return dict(kind=kind, field=rng.choice(["nacl", "fcc"]), storage=rng.choice(["f32", "f16", "bf16"]),
                    replicas=log_int(16, 1600000 // atoms if kind == "relax_rigid" else 4096), atoms=atoms, steps=rng.randint(40, 50))
    atoms = rng.choice([0, log_int(5, 120)])       # 0: the uneven batch
    most = {"relax_flex": 16384, "run_flex": 2048, "langevin": 5000, "eval": 16384}[kind]
    c = dict(kind=kind, field=rng.choice(["nacl", "hard"]), storage="f32", replicas=log_int(16, most), atoms=atoms)
    if kind != "eval":
        c["steps"] = {"relax_flex": rng.randint(8, 16), "run_flex": rng.randint(6, 10), "langevin": rng.randint(10, 20)}[kind]
    return c


# ---------------------------------------------------------------------------
# inputs: substrates, molecules, starts
# ---------------------------------------------------------------------------
@functools.lru_cache(None)
def context():
    """The library context that a program keeps."""
    return G.Context(0)


@functools.lru_cache(None)
def substrate(field):
    if field == "fcc":
        return synth.fcc111_slab(a=4.08, ncell=12, layers=4)
    morse = synth.HARD_CATION if field == "hard" else None
    return synth.rocksalt_slab(a=5.64, ncell=8, layers=3, charge=0.7, cation_morse=morse)


def ghosts(spacing):
    """Node planes below the floor: 8 at 0.1 A as in the benchmark, fewer on coarser grids (they stay above the slab)."""
    return min(8, int(0.8 / spacing + 1e-9))


@functools.lru_cache(None)
def grid_of(field, storage):
    """The substrate's grid at 0.1 A, built once and kept."""
    sub = substrate(field)
    box = synth.grid_box_for(sub, 0.1, height=20.0)
    return G.build_grid(context(), sub, box.origin, box.length, box.spacing, storage=STORE[storage],
                        ghost_below=ghosts(0.1))


@functools.lru_cache(None)
def molecule(kind, atoms):
    if kind == "rigid":
        return (synth.c24h8o6_core() if atoms == 38 else synth.rigid_molecule(atoms, 2024))
    return synth.random_flexible_molecule(atoms, 4, 2222)


@functools.lru_cache(None)
def uneven_templates():
    """64 molecules of 10 to 120 atoms (log-uniform) with up to 12 torsion bonds."""
    return synth.uneven_batch(1, 64, 77)[0]


def _rng(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _rotations(n, g):
    q = torch.randn(n, 4, generator=g, device=DEV, dtype=torch.float64)
    q = q / q.norm(dim=1, keepdim=True)
    return q, _matrices(q)


def _matrices(q):
    w, x, y, z = q.unbind(-1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], -1).reshape(*q.shape[:-1], 3, 3)


def _centres(sub, lowest, g, clear):
    """Centres over the tile, 3 to 5 A above the top layer, raised until the lowest atom keeps `clear`."""
    u = torch.rand(len(lowest), 3, generator=g, device=DEV, dtype=torch.float64)
    c = torch.stack([u[:, 0] * sub.tile[0], u[:, 1] * sub.tile[1], sub.z_top + 3.0 + 2.0 * u[:, 2]], 1)
    c[:, 2] += (sub.z_top + clear - (c[:, 2] + lowest)).clamp_min(0.0)
    return c


def rigid_start(case, seed):
    """Poses (n, 7) and 300 K velocities (n, 6) of a batch of one rigid molecule."""
    mol, sub, n, g = molecule("rigid", case["atoms"]), substrate(case["field"]), case["replicas"], _rng(seed)
    body = torch.tensor(mol.xyz, device=DEV)
    q, R = _rotations(n, g)
    c = _centres(sub, (R[:, 2] @ body.T).amin(1), g, 2.0)
    M, I = _inertia(mol)
    sd = torch.sqrt(KB * 300.0 * ACC / torch.cat([M.expand(3), I]))
    v = torch.randn(n, 6, generator=g, device=DEV, dtype=torch.float64) * sd
    return torch.cat([c, q], 1).float().contiguous(), v.float().contiguous()


def flexible_batch(case):
    """(templates, template of every replica)."""
    if case["atoms"]:
        return (molecule("flexible", case["atoms"]),), np.zeros(case["replicas"], np.int32)
    t = uneven_templates()
    return tuple(t), np.random.default_rng(77).integers(0, len(t), case["replicas"]).astype(np.int32)


def flexible_start(case, seed):
    """Positions and 300 K velocities (atoms of all replicas, 3), bonds off their rest lengths as in a running simulation."""
    mols, tof = flexible_batch(case)
    sub, g, n = substrate(case["field"]), _rng(seed), len(tof)
    most = max(m.n for m in mols)
    ref = torch.zeros(len(mols), most, 3, device=DEV, dtype=torch.float64)
    mass = torch.ones(len(mols), most, device=DEV, dtype=torch.float64)
    live = torch.zeros(len(mols), most, device=DEV, dtype=torch.bool)
    for k, m in enumerate(mols):
        ref[k, :m.n] = torch.tensor(m.xyz - m.xyz.mean(0), device=DEV)
        mass[k, :m.n] = torch.tensor(m.mass, device=DEV)
        live[k, :m.n] = True
    t = torch.tensor(tof, device=DEV, dtype=torch.long)
    _, R = _rotations(n, g)
    x = torch.einsum("nij,naj->nai", R, ref[t])
    x = x + 0.02 * torch.randn(x.shape, generator=g, device=DEV, dtype=torch.float64)
    low = torch.where(live[t], x[:, :, 2], torch.inf).amin(1)
    x = x + _centres(sub, low, g, 3.0 if case["field"] == "hard" else 2.0)[:, None]
    v = torch.randn(x.shape, generator=g, device=DEV, dtype=torch.float64) * torch.sqrt(KB * 300.0 * ACC / mass[t])[..., None]
    return x[live[t]].float().contiguous(), v[live[t]].float().contiguous()


def point_inputs(case, seed):
    """Points over the tile, 2 to 8 A above the floor, with the grid factors (Q, P, L) of C, H and O atoms."""
    sub, g, n = substrate(case["field"]), _rng(seed), case["points"]
    box = synth.grid_box_for(sub, 0.1, height=20.0)
    u = torch.rand(n, 3, generator=g, device=DEV, dtype=torch.float64)
    lo = torch.tensor([0.0, 0.0, box.origin[2] + 2.0], device=DEV, dtype=torch.float64)
    x = lo + u * torch.tensor([box.length[0], box.length[1], 6.0], device=DEV, dtype=torch.float64)
    el = torch.tensor([synth.ELEMENTS[e][:2] for e in ("C", "H", "O")], device=DEV, dtype=torch.float64)
    R, eps = el[torch.randint(0, 3, (n,), generator=g, device=DEV)].unbind(1)
    q = 0.6 * torch.rand(n, generator=g, device=DEV, dtype=torch.float64) - 0.3
    f = torch.stack([q, eps * torch.exp(2 * ALPHA * R), -2 * eps * torch.exp(ALPHA * R)], 1)
    return x.float().contiguous(), f.float().contiguous()


def train_inputs(case, seed):
    """Initial weights, 4096 target poses, the molecule's descriptor and the loop's seed."""
    r = np.random.default_rng(seed)
    Ws, bs = synth.mlp_weights(NET, int(seed) % (1 << 31))
    T = np.zeros((4096, 19), np.float32)
    T[:, :2] = r.uniform(0.0, 5.64, (4096, 2))
    T[:, 2] = r.uniform(8.5, 9.5, 4096)
    q = r.standard_normal((4096, 4))
    T[:, 3:7] = q / np.linalg.norm(q, axis=1, keepdims=True)
    T[:, 7:] = r.uniform(-math.pi, math.pi, (4096, 12))
    mask = (r.random((4096, 12)) < 0.5).astype(np.float32)
    desc = np.zeros(64, np.float32)
    desc[:14] = r.uniform(0.0, 1.0, 14)
    return [W.astype(np.float32) for W in Ws], [b.astype(np.float32) for b in bs], T, mask, desc, int(seed) * 2 + 1


# ---------------------------------------------------------------------------
# the library's side
# ---------------------------------------------------------------------------
def _out(n, dtype=torch.float32):
    return torch.empty(n, dtype=dtype, device=DEV)


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case, ctx=context())
    if kind == "train":
        Ws, bs, T, mask, s["desc"], s["seed"] = train_inputs(case, seed)
        s["net"] = G.MLP(s["ctx"], NET)
        s["net"].set_params(Ws, bs)
        s["net"].set_targets(T, mask)
        s["params"] = G.train_params(lr=1e-3, tile=(5.64, 5.64))
        return s
    if kind == "build":
        # the charge and the Morse parameters of this substrate, as another material would have them
        f = np.random.default_rng(seed).uniform(0.9, 1.1, 3)
        sub = build_substrate(case, f)
        s["sub"], s["box"] = sub, synth.grid_box_for(sub, case["spacing"], height=20.0)
        return s
    s["grid"] = grid_of(case["field"], case["storage"])
    if kind == "points":
        s["x"], s["f"] = point_inputs(case, seed)
        n = case["points"]
        s["out"] = (_out(n), _out((n, 3)), _out(n, torch.int32))
        return s
    if kind in ("relax_rigid", "run_rigid"):
        s["x"], s["v"] = rigid_start(case, seed)
        s["reps"] = G.Replicas(s["ctx"], [molecule("rigid", case["atoms"])], np.zeros(case["replicas"], np.int32), rigid=True)
    else:
        mols, tof = flexible_batch(case)
        s["x"], s["v"] = flexible_start(case, seed)
        s["reps"] = G.Replicas(s["ctx"], list(mols), tof)
    s["fire"] = G.fire_params(f_conv=1e-3)
    n, na = case["replicas"], s["reps"].n_atoms
    s["ox"], s["ov"], s["oe"] = _out(s["x"].shape), _out(s["v"].shape), _out(n, torch.float64)
    s["st"], s["steps"] = _out(n, torch.int32), _out(n, torch.int32)
    if kind == "eval":
        s["out"] = (s["oe"], _out((na, 3)), _out(na), s["st"])
        s["reps"].set_state(s["x"])
    return s


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "train":
        net = s["net"]
        losses = net.train(case["steps"], case["targets"], case["proposals"], s["desc"], s["seed"], s["params"])
        return {"losses": losses, "weights": net.get_params()[0]}
    if kind == "build":
        g = G.build_grid(ctx, s["sub"], s["box"].origin, s["box"].length, s["box"].spacing, keep_f64=True,
                         ghost_below=ghosts(s["box"].spacing))
        c = g.download_f64("coefs")
        g.close()
        return {"C": c[0], "P": c[1], "L": c[2]}
    grid = s["grid"]
    if kind == "points":
        E, F, S = G.eval_points(ctx, grid, s["x"], s["f"], out=s["out"], flags=G.POINTS_BINNED if case["binned"] else 0)
        return {"E": E, "F": F, "status": S}
    reps = s["reps"]
    if kind == "eval":
        E, F, Ea, S = G.eval(ctx, grid, reps, out=s["out"])
        return {"E": E.float(), "F": F, "E_atom": Ea, "status": S}
    dynamics = kind in ("run_rigid", "run_flex", "langevin")
    reps.set_state(s["x"], s["v"] if dynamics else None, flags=G.ASYNC)
    trace = None
    if kind == "langevin":
        G.langevin(ctx, grid, reps, case["steps"], 1.0, 300.0, 0.01, seed=12345)
    elif dynamics:
        _, trace = G.run(ctx, grid, reps, case["steps"], 1.0, record_every=5)
    else:
        G.relax(ctx, grid, reps, case["steps"], s["fire"])
    ctx.check(G.lib.gridff_get_state(reps.h, _p(s["ox"]), _p(s["ov"]), G.DEVICE_PTRS | G.ASYNC))
    ctx.check(G.lib.gridff_get_fire_state(reps.h, None, None, None, _p(s["st"]), _p(s["steps"]), _p(s["oe"]), G.DEVICE_PTRS))
    out = {"x": s["ox"], "v": s["ov"], "E": s["oe"].float(), "status": s["st"]}
    if trace is not None:
        out["trace"] = trace.astype(np.float32)
    if not dynamics:
        out["steps"] = s["steps"]
    return out


def work(case):
    """Bytes: state in and out, parameters, and the grid nodes that a first evaluation touches.  Flops: per atom and
    evaluation 64 nodes x (channel combination 5 + value and gradient 6), per pair 40, per bonded term 60."""
    kind = case["kind"]
    if kind == "train":
        rows = case["targets"] * case["proposals"]
        macs = sum(a * b for a, b in zip(NET[:-1], NET[1:]))
        return {"bytes": 4 * 4 * macs * 1.0 + 4 * 4096 * 31, "flops": 6.0 * rows * macs * case["steps"]}
    if kind == "build":
        sub = build_substrate(case, np.ones(3))
        n = [math.ceil(L / case["spacing"] - 1e-9) for L in (*sub.tile, 20.0)]
        nodes = n[0] * n[1] * (n[2] + ghosts(case["spacing"]))
        # the Morse sums: every atom of the slab within the cutoff of a node, averaged over the box height
        near = sub.n / abs(float(np.linalg.det(sub.cell[:2, :2]))) * math.pi * RCUT * RCUT / 2
        return {"bytes": nodes * (3 * 8.0 + 16.0), "flops": nodes * near * 40.0}
    node = 12 if case["storage"] == "f32" else 6
    if kind == "points":
        n = case["points"]
        return {"bytes": n * (24 + 20.0) + min(n * 64 * node, 2.7e6 * node), "flops": n * 704.0}
    steps = case.get("steps", 0) + (kind != "relax_flex" and kind != "relax_rigid")
    if kind in ("relax_rigid", "run_rigid"):
        n, at = case["replicas"], case["replicas"] * case["atoms"]
        return {"bytes": n * 2 * 52.0 + min(at * 64 * node, 2.7e6 * node), "flops": at * steps * 704.0}
    sizes = [case["atoms"]] if case["atoms"] else [m.n for m in uneven_templates()]
    at = case["replicas"] * sum(sizes) / len(sizes)
    pairs = case["replicas"] * sum(k * (k - 1) / 2 for k in sizes) / len(sizes)
    return {"bytes": at * 48.0 + min(at * 64 * node, 2.7e6 * node), "flops": steps * (at * (704.0 + 3 * 60) + pairs * 40.0)}


def build_substrate(case, factors):
    s = synth.rocksalt_slab(a=5.64, ncell=case["cells"], layers=case["layers"], charge=0.7 * float(factors[0]))
    s.R, s.eps = s.R * float(factors[1]), s.eps * float(factors[2])
    return s


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
def _d(a):
    """The FP32 values that the library is given, in 64 bits."""
    if not isinstance(a, torch.Tensor):
        a = torch.tensor(np.asarray(a))
    return a.to(DEV).float().double()


def _coefficients(sub, box, coulomb):
    """(coefficients (C, P, L) in 64 bits, origin, spacing) of the grid over `box` with its ghost planes."""
    n = [math.ceil(L / box.spacing - 1e-9) for L in box.length]
    h = [L / k for L, k in zip(box.length, n)]
    below = ghosts(box.spacing)
    n[2] += below
    org = [box.origin[0], box.origin[1], box.origin[2] - below * h[2]]
    ax = [torch.arange(n[a], device=DEV, dtype=torch.float64) * h[a] + org[a] for a in range(3)]
    # lattice images whose atoms come within the cutoff of the box
    A = sub.cell[:2, :2]
    reach = RCUT + math.hypot(*box.length[:2])
    k = int(math.ceil((reach + np.abs(sub.xyz[:, :2]).max()) / min(abs(np.linalg.det(A)) / np.linalg.norm(A, axis=1)))) + 1
    P, ids = [], []
    for i in range(-k, k + 1):
        for j in range(-k, k + 1):
            p = sub.xyz + np.array([*(i * A[0] + j * A[1]), 0.0])
            gap = np.maximum(0.0, np.maximum(np.array(box.origin[:2]) - p[:, :2], p[:, :2] - np.array(box.origin[:2]) - np.array(box.length[:2])))
            near = (gap ** 2).sum(1) < RCUT ** 2
            P.append(p[near])
            ids.append(np.nonzero(near)[0])
    P, ids = torch.tensor(np.concatenate(P), device=DEV), np.concatenate(ids)
    R, eps = torch.tensor(sub.R[ids], device=DEV), torch.tensor(sub.eps[ids], device=DEV)
    vals = torch.zeros(3, *n, device=DEV, dtype=torch.float64)
    dz2 = (ax[2][:, None] - P[:, 2]) ** 2
    for i in range(n[0]):
        for j0 in range(0, n[1], 32):
            d2 = ((ax[0][i] - P[:, 0]) ** 2 + (ax[1][j0:j0 + 32, None] - P[:, 1]) ** 2)[:, None] + dz2
            e = torch.where(d2 < RCUT ** 2, torch.exp(-ALPHA * (torch.sqrt(d2) - R)), 0.0)
            vals[2, i, j0:j0 + 32] = e @ eps
            vals[1, i, j0:j0 + 32] = (e * e) @ eps
    if coulomb:
        vals[0] = _slab_potential(sub, ax)
    # exact cubic B-spline fit: periodic along x and y, the end coefficient repeated along z
    for a in (0, 1):
        f = (2.0 + torch.cos(2 * math.pi * torch.arange(n[a], device=DEV, dtype=torch.float64) / n[a])) / 3.0
        f = f.reshape([-1 if d == a + 1 else 1 for d in range(4)])
        vals = torch.fft.ifft(torch.fft.fft(vals, dim=a + 1) / f, dim=a + 1).real
    m = torch.diag(torch.full((n[2],), 2 / 3, device=DEV, dtype=torch.float64))
    o = torch.full((n[2] - 1,), 1 / 6, device=DEV, dtype=torch.float64)
    m = m + torch.diag(o, 1) + torch.diag(o, -1)
    m[0, 0] = m[-1, -1] = 5 / 6
    vals = torch.linalg.solve(m, vals.reshape(-1, n[2]).T).T.reshape(3, *n)
    return vals, org, h


def _slab_potential(sub, ax):
    """Potential (V) above a slab of square neutral layers of period 5.64 A: sum over the layers' reciprocal vectors."""
    a = 5.64
    fold = np.concatenate([np.mod(sub.xyz[:, :2] + 1e-7, a) - 1e-7, sub.xyz[:, 2:], sub.q[:, None]], 1)
    cell = fold[np.unique(np.round(fold[:, :3], 6), axis=0, return_index=True)[1]]
    clear = float(ax[2][0]) - sub.z_top
    m = int(32.0 / clear * a / (2 * math.pi)) + 1
    k = 2 * math.pi / a * torch.arange(-m, m + 1, device=DEV, dtype=torch.float64)
    gx, gy = k[:, None], k[None, :]
    gn = torch.sqrt(gx * gx + gy * gy)
    inv = torch.where(gn > 0, 2 * math.pi / (a * a) / gn.clamp_min(1e-300), 0.0)
    # the layers' structure factors, moved to the height of the first node plane
    S = sum(float(q) * torch.exp(-1j * (gx * float(u) + gy * float(w)) - gn * (ax[2][0] - float(z))) for u, w, z, q in cell)
    ex = torch.exp(1j * ax[0][:, None] * k)
    ey = torch.exp(1j * ax[1][:, None] * k)
    out = torch.empty(len(ax[0]), len(ax[1]), len(ax[2]), device=DEV, dtype=torch.float64)
    for l, z in enumerate(ax[2]):
        out[:, :, l] = (ex @ (S * inv * torch.exp(-gn * (z - ax[2][0]))) @ ey.T).real
    return KE * out


class _Field:
    """The tricubic field of a grid in 64 bits, from the coefficients as the storage holds them."""

    def __init__(self, field, storage):
        sub = substrate(field)
        box = synth.grid_box_for(sub, 0.1, height=20.0)
        c, self.org, self.h = _coefficients(sub, box, bool(np.any(sub.q != 0)))
        if storage == "f32":
            c = c.float().double()
        else:
            for k in range(3):
                e = math.frexp(float(c[k].abs().max()))[1]
                c[k] = (c[k] * 2.0 ** (15 - e)).to(torch.float16 if storage == "f16" else torch.bfloat16).double() * 2.0 ** (e - 15)
        self.n = c.shape[1:]
        self.c = c.permute(1, 2, 3, 0).reshape(-1, 3).contiguous()

    def __call__(self, x, f):
        """(energy, force) of points x (n, 3) with factors f (n, 3)."""
        E, F = [], []
        for a in range(0, len(x), 400000):
            e, g = self._part(x[a:a + 400000], f[a:a + 400000])
            E.append(e)
            F.append(g)
        return torch.cat(E), torch.cat(F)

    def _part(self, x, f):
        W, D, I = [], [], []
        o = torch.arange(-1, 3, device=DEV)
        for a in range(3):
            u = (x[:, a] - self.org[a]) / self.h[a]
            if a == 2:
                inside = u < self.n[2] - 1
                u = u.clamp(0.0, self.n[2] - 1.0)
            i = torch.floor(u)
            t = (u - i)[:, None]
            s = 1 - t
            W.append(torch.cat([s ** 3 / 6, (4 - 6 * t ** 2 + 3 * t ** 3) / 6, (4 - 6 * s ** 2 + 3 * s ** 3) / 6, t ** 3 / 6], 1))
            D.append(torch.cat([-s ** 2 / 2, 1.5 * t ** 2 - 2 * t, 2 * s - 1.5 * s ** 2, t ** 2 / 2], 1) / self.h[a])
            j = i.long()[:, None] + o
            I.append(j.clamp(0, self.n[2] - 1) if a == 2 else j % self.n[a])
        at = ((I[0][:, :, None, None] * self.n[1] + I[1][:, None, :, None]) * self.n[2] + I[2][:, None, None, :])
        c = (self.c[at.reshape(len(x), -1)] @ f[:, :, None]).reshape(len(x), 4, 4, 4)
        c = torch.where(inside[:, None, None, None], c, 0.0)
        con = lambda p, q, r: torch.einsum("nabc,na,nb,nc->n", c, p, q, r)  # noqa: E731
        return con(*W), -torch.stack([con(D[0], W[1], W[2]), con(W[0], D[1], W[2]), con(W[0], W[1], D[2])], 1)


@functools.lru_cache(None)
def field_of(field, storage):
    return _Field(field, storage)


def _factors(mol):
    q, R, eps = _d(mol.q), _d(mol.R), _d(mol.eps)
    return torch.stack([q, eps * torch.exp(2 * ALPHA * R), -2 * eps * torch.exp(ALPHA * R)], 1)


def _inertia(mol):
    m, b = _d(mol.mass), _d(mol.xyz)
    return m.sum(), torch.stack([(m * (b[:, (k + 1) % 3] ** 2 + b[:, (k + 2) % 3] ** 2)).sum() for k in range(3)])


class _Rigid:
    def __init__(self, case):
        self.mol = molecule("rigid", case["atoms"])
        self.body, self.f = _d(self.mol.xyz), _factors(self.mol)
        self.M, self.I = _inertia(self.mol)
        self.rmax = float(self.body.norm(dim=1).max())
        self.field = field_of(case["field"], case["storage"])

    def forces(self, c, q):
        """(energy, total force, body-frame torque)."""
        R = _matrices(q)
        arm = torch.einsum("nij,aj->nai", R, self.body)
        E, F = self.field((arm + c[:, None]).reshape(-1, 3), self.f.repeat(len(c), 1))
        F = F.reshape(arm.shape)
        tau = torch.linalg.cross(arm, F).sum(1)
        return E.reshape(len(c), -1).sum(1), F.sum(1), torch.einsum("nij,ni->nj", R, tau)


def _quat_mul(a, b):
    w, x, y, z = a.unbind(1)
    s, t, u, v = b.unbind(1)
    return torch.stack([w * s - x * t - y * u - z * v, w * t + x * s + y * v - z * u,
                        w * u - x * v + y * s + z * t, w * v + x * u - y * t + z * s], 1)


def _fire_scalars(n):
    return dict(dt=torch.full((n, 1), 0.5, device=DEV, dtype=torch.float64), al=torch.full((n, 1), 0.1, device=DEV, dtype=torch.float64),
                np=torch.zeros(n, 1, device=DEV))


def _fire_decide(s, up):
    """FIRE's step and mixing after the power test; the caller mixes with the returned old mixing."""
    old = s["al"]
    grow = up & (s["np"] > 5)
    s["dt"] = torch.where(grow, (s["dt"] * 1.1).clamp_max(2.0), torch.where(up, s["dt"], s["dt"] * 0.5))
    s["al"] = torch.where(grow, s["al"] * 0.99, torch.where(up, s["al"], 0.1))
    s["np"] = torch.where(up, s["np"] + 1, 0)
    return old


def _unit(a):
    n = a.norm(dim=1, keepdim=True)
    return torch.where(n > 0, a / n.clamp_min(1e-300), 0.0), n


def _relax_rigid(case, seed):
    r = _Rigid(case)
    x, _ = rigid_start(case, seed)
    c, q = x[:, :3].double(), x[:, 3:].double()
    v, w = torch.zeros_like(c), torch.zeros_like(c)
    s, E = _fire_scalars(len(c)), None
    go = torch.ones(len(c), 1, device=DEV, dtype=torch.bool)
    for _ in range(case["steps"]):
        e, F, T = r.forces(c, q)
        E = e if E is None else torch.where(go[:, 0], e, E)
        go = go & ((F * F + T * T).sum(1, keepdim=True) >= 1e-6)
        keep = {k: s[k] for k in s}
        up = (F * v + T * w).sum(1, keepdim=True) > 0
        a = _fire_decide(s, up)
        Fh, _ = _unit(F)
        Th, _ = _unit(T)
        nv = torch.where(up, (1 - a) * v + a * v.norm(dim=1, keepdim=True) * Fh, 0.0) + ACC * s["dt"] * F / r.M
        nw = torch.where(up, (1 - a) * w + a * w.norm(dim=1, keepdim=True) * Th, 0.0) + ACC * s["dt"] * T / r.I
        dr = nv * s["dt"]
        dr = dr * (0.1 / dr.norm(dim=1, keepdim=True).clamp_min(1e-300)).clamp_max(1.0)
        u, wn = _unit(nw)
        half = 0.5 * (wn * s["dt"]).clamp_max(0.1 / r.rmax)
        nq = _quat_mul(q, torch.cat([torch.cos(half), torch.sin(half) * u], 1))
        nq = nq / nq.norm(dim=1, keepdim=True)
        c, q, v, w = (torch.where(go, b, o) for b, o in ((c + dr, c), (nq, q), (nv, v), (nw, w)))
        s = {k: torch.where(go, s[k], keep[k]) for k in s}
    return {"x": torch.cat([c, q], 1), "v": torch.cat([v, w], 1), "E": E, "status": None, "steps": None}


def _run_rigid(case, seed):
    """The NO_SQUISH splitting with the quaternion's conjugate momentum p = 2 q (0, L)."""
    r = _Rigid(case)
    x, v6 = rigid_start(case, seed)
    c, q, v, om = x[:, :3].double(), x[:, 3:].double(), v6[:, :3].double(), v6[:, 3:].double()
    zero = torch.zeros(len(c), 1, device=DEV, dtype=torch.float64)
    conj = torch.tensor([1.0, -1.0, -1.0, -1.0], device=DEV, dtype=torch.float64)
    unit = torch.eye(4, device=DEV, dtype=torch.float64)
    p = 2 * _quat_mul(q, torch.cat([zero, om * r.I], 1))

    def spin():
        return 0.5 * _quat_mul(q * conj, p)[:, 1:]

    def total(e):
        L = spin()
        return e + 0.5 * (r.M * (v * v).sum(1) + (L * L / r.I).sum(1)) / ACC

    e, F, T = r.forces(c, q)
    trace = [total(e)]
    for k in range(case["steps"]):
        v = v + 0.5 * ACC * F / r.M
        p = p + ACC * _quat_mul(q, torch.cat([zero, T], 1))
        c = c + v
        for axis, h in ((3, 0.5), (2, 0.5), (1, 1.0), (2, 0.5), (3, 0.5)):
            b = unit[axis].expand(len(c), 4)
            pq, pp = _quat_mul(q, b), _quat_mul(p, b)
            z = h * (p * pq).sum(1, keepdim=True) / (4 * r.I[axis - 1])
            q, p = torch.cos(z) * q + torch.sin(z) * pq, torch.cos(z) * p + torch.sin(z) * pp
        e, F, T = r.forces(c, q)
        v = v + 0.5 * ACC * F / r.M
        p = p + ACC * _quat_mul(q, torch.cat([zero, T], 1))
        if (k + 1) % 5 == 0:
            trace.append(total(e))
    return {"x": torch.cat([c, q], 1), "v": torch.cat([v, spin() / r.I], 1), "E": e, "status": None, "trace": torch.stack(trace)}


class _Flexible:
    """All replicas' terms as flat index lists; forces by differentiating the energy."""

    def __init__(self, case, seed):
        mols, tof = flexible_batch(case)
        sizes = np.array([m.n for m in mols])[tof]
        off = np.concatenate([[0], np.cumsum(sizes)])
        self.n_rep, self.rep = len(tof), torch.tensor(np.repeat(np.arange(len(tof)), sizes), device=DEV)
        parts = {k: [] for k in ("bond", "angle", "tors", "pair")}
        self.f = torch.cat([_factors(m) for m in mols])
        start = np.concatenate([[0], np.cumsum([m.n for m in mols])])
        take = torch.tensor(np.concatenate([start[t] + np.arange(mols[t].n) for t in tof]), device=DEV)
        self.f = self.f[take]
        self.mass = torch.cat([_d(m.mass) for m in mols])[take][:, None]
        self.q, self.R, self.eps = (torch.cat([_d(getattr(m, k)) for m in mols])[take] for k in ("q", "R", "eps"))
        for t, m in enumerate(mols):
            o = off[:-1][tof == t]
            if not len(o):
                continue
            near = np.eye(m.n, dtype=bool)
            near[m.bonds[:, 0], m.bonds[:, 1]] = near[m.bonds[:, 1], m.bonds[:, 0]] = True
            near = (near.astype(np.int64) @ near.astype(np.int64)) > 0      # at most two bonds apart
            pairs = np.argwhere(np.triu(~near, 1))
            for key, idx, prm in (("bond", m.bonds, (m.bond_k, m.bond_r0)), ("angle", m.angles, (m.angle_k, m.angle_cos0)),
                                  ("tors", m.torsions, (m.torsion_V, m.torsion_n, m.torsion_cos_nphi0)), ("pair", pairs, ())):
                if len(idx):
                    parts[key].append(((o[:, None, None] + idx[None]).reshape(-1, idx.shape[1]), [np.tile(np.asarray(p, np.float64), len(o)) for p in prm]))
        self.terms = {}
        for key, ps in parts.items():
            if ps:
                idx = torch.tensor(np.concatenate([p[0] for p in ps]), device=DEV).long().T.contiguous()
                self.terms[key] = (idx, [_d(np.concatenate(c)) for c in zip(*[p[1] for p in ps])])
        self.field = field_of(case["field"], case["storage"])

    def intra(self, x):
        x = x.detach().requires_grad_(True)
        E = torch.zeros(self.n_rep, device=DEV, dtype=torch.float64)
        for key, (i, prm) in self.terms.items():
            if key == "bond":
                e = prm[0] * ((x[i[0]] - x[i[1]]).norm(dim=1) - prm[1]) ** 2
            elif key == "angle":
                u, w = x[i[0]] - x[i[1]], x[i[2]] - x[i[1]]
                e = prm[0] * ((u * w).sum(1) / (u.norm(dim=1) * w.norm(dim=1)) - prm[1]) ** 2
            elif key == "tors":
                b1, b2, b3 = x[i[1]] - x[i[0]], x[i[2]] - x[i[1]], x[i[3]] - x[i[2]]
                n1, n2 = torch.linalg.cross(b1, b2), torch.linalg.cross(b2, b3)
                phi = torch.atan2(b2.norm(dim=1) * (b1 * n2).sum(1), (n1 * n2).sum(1))
                e = 0.5 * prm[0] * (1 - prm[2] * torch.cos(prm[1] * phi))
            else:
                r = (x[i[0]] - x[i[1]]).norm(dim=1)
                m = torch.exp(-ALPHA * (r - self.R[i[0]] - self.R[i[1]]))
                e = self.eps[i[0]] * self.eps[i[1]] * m * (m - 2) + KE * self.q[i[0]] * self.q[i[1]] / r
            E = E.index_add(0, self.rep[i[0]], e)
        (g,) = torch.autograd.grad(E.sum(), x) if self.terms else (torch.zeros_like(x),)
        return E.detach(), -g

    def sums(self, a):
        return torch.zeros(self.n_rep, device=DEV, dtype=torch.float64).index_add(0, self.rep, a)

    def forces(self, x):
        """(energy per replica, forces, grid energy per atom)."""
        Eg, Fg = self.field(x, self.f)
        Ei, Fi = self.intra(x)
        return Ei + self.sums(Eg), Fg + Fi, Eg


def _relax_flexible(case, seed):
    m = _Flexible(case, seed)
    x = flexible_start(case, seed)[0].double()
    v = torch.zeros_like(x)
    s, E = _fire_scalars(m.n_rep), None
    go = torch.ones(m.n_rep, 1, device=DEV, dtype=torch.bool)
    for _ in range(case["steps"]):
        e, F, _ = m.forces(x)
        E = e if E is None else torch.where(go[:, 0], e, E)
        f2 = m.sums((F * F).sum(1))[:, None]
        go = go & (f2 >= 1e-6)
        keep = {k: s[k] for k in s}
        up = m.sums((F * v).sum(1))[:, None] > 0
        a = _fire_decide(s, up)
        mix = a * torch.sqrt(m.sums((v * v).sum(1))[:, None] / f2)
        up, a, mix, dt = (t[m.rep] for t in (up, a, mix, s["dt"]))
        nv = torch.where(up, (1 - a) * v + mix * F, 0.0) + ACC * dt * F / m.mass
        d = nv * dt
        d = d * (0.1 / d.norm(dim=1, keepdim=True).clamp_min(1e-300)).clamp_max(1.0)
        live = go[m.rep]
        x, v = torch.where(live, x + d, x), torch.where(live, nv, v)
        s = {k: torch.where(go, s[k], keep[k]) for k in s}
    return {"x": x, "v": v, "E": E, "status": None, "steps": None}


def _splitmix(x):
    with np.errstate(over="ignore"):
        x = x + np.uint64(0x9E3779B97F4A7C15)
        x = (x ^ (x >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return x ^ (x >> np.uint64(31))


def _normals(s):
    u1 = ((s >> np.uint64(40)).astype(np.float64) + 1) / 2.0 ** 24
    u2 = ((s >> np.uint64(16)) & np.uint64(0xFFFFFF)).astype(np.float64) / 2.0 ** 24
    return np.sqrt(-2 * np.log(u1)) * np.cos(2 * np.pi * u2)


def _dynamics(case, seed):
    """Velocity Verlet, or its BAOAB form at 300 K and friction 0.01 / fs with the library's counter-based noise."""
    m = _Flexible(case, seed)
    x, v = (a.double() for a in flexible_start(case, seed))
    heat = case["kind"] == "langevin"
    c1 = math.exp(-0.01) if heat else 1.0
    if heat:
        rep = m.rep.cpu().numpy()
        first = np.searchsorted(rep, np.arange(m.n_rep))
        comp = (3 * (np.arange(len(rep)) - first[rep]))[:, None] + np.arange(3)
        key = _splitmix(np.uint64(12345) ^ _splitmix(rep.astype(np.uint64)))[:, None]

    def total(e):
        return e + m.sums(0.5 * (m.mass * v * v).sum(1)) / ACC

    e, F, _ = m.forces(x)
    trace = [total(e)]
    for k in range(case["steps"]):
        v = v + 0.5 * ACC * F / m.mass
        x = x + 0.5 * v
        if heat:
            xi = torch.tensor(_normals(_splitmix(key ^ (np.uint64(512 * k) + comp.astype(np.uint64)))), device=DEV)
            v = c1 * v + math.sqrt(1 - c1 * c1) * torch.sqrt(KB * 300.0 * ACC / m.mass) * xi
        x = x + 0.5 * v
        e, F, _ = m.forces(x)
        v = v + 0.5 * ACC * F / m.mass
        if (k + 1) % 5 == 0:
            trace.append(total(e))
    out = {"x": x, "v": v, "E": e, "status": None}
    if not heat:
        out["trace"] = torch.stack(trace)
    return out


def _train(case, seed):
    """The training loop in 64 bits throughout (the library rounds the operands of its products to bfloat16)."""
    Ws, bs, T, mask, desc, loop = train_inputs(case, seed)
    prm = [p for W, b in zip(Ws, bs) for p in (_d(W).requires_grad_(True), _d(b).requires_grad_(True))]
    B, K, n_noise = case["targets"], case["proposals"], NET[0] - len(desc)
    mom = [[torch.zeros_like(p), torch.zeros_like(p)] for p in prm]
    T, mask, tile = _d(T), _d(mask), 5.64
    losses = []
    loop = np.uint64(loop)
    for k in range(case["steps"]):
        row = _splitmix(loop ^ _splitmix(np.uint64(k << 20) + np.arange(B, dtype=np.uint64))) % np.uint64(len(T))
        row = torch.tensor(row.astype(np.int64), device=DEV)
        ctr = ((np.uint64(k << 20) + np.arange(B * K, dtype=np.uint64)) << np.uint64(6))[:, None] + np.arange(n_noise, dtype=np.uint64)
        h = torch.cat([_d(desc).expand(B * K, -1), torch.tensor(_normals(_splitmix(loop ^ _splitmix(ctr))), device=DEV)], 1)
        for l in range(len(NET) - 1):
            h = h @ prm[2 * l].T + prm[2 * l + 1]
            h = torch.relu(h) if l < len(NET) - 2 else h
        o, t, m = h.reshape(B, K, 19), T[row][:, None], mask[row][:, None]
        dc = o[..., :3] - t[..., :3]
        dc = torch.cat([dc[..., :2] - tile * torch.round(dc[..., :2] / tile).detach(), dc[..., 2:]], -1)
        s = (o[..., 3:7] / o[..., 3:7].norm(dim=-1, keepdim=True) * t[..., 3:7]).sum(-1)
        d = (dc * dc).sum(-1) + 1 - s * s + 0.25 * (m * (1 - torch.cos(o[..., 7:] - t[..., 7:]))).sum(-1)
        loss = d.amin(1).mean()
        losses.append(loss.detach())
        for p, g, mv in zip(prm, torch.autograd.grad(loss, prm), mom):
            mv[0] = 0.9 * mv[0] + 0.1 * g
            mv[1] = 0.999 * mv[1] + 0.001 * g * g
            with torch.no_grad():
                p -= 1e-3 / (1 - 0.9 ** (k + 1)) * mv[0] / (torch.sqrt(mv[1] / (1 - 0.999 ** (k + 1))) + 1e-8)
    return {"losses": torch.stack(losses), "weights": torch.cat([p.detach().reshape(-1) for p in prm])}


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _train(case, seed)
    if kind == "build":
        sub = build_substrate(case, np.random.default_rng(seed).uniform(0.9, 1.1, 3))
        c, _, _ = _coefficients(sub, synth.grid_box_for(sub, case["spacing"], height=20.0), True)
        return {"C": c[0], "P": c[1], "L": c[2]}
    if kind == "points":
        x, f = point_inputs(case, seed)
        E, F = field_of(case["field"], case["storage"])(x.double(), f.double())
        return {"E": E, "F": F, "status": None}
    if kind == "relax_rigid":
        return _relax_rigid(case, seed)
    if kind == "run_rigid":
        return _run_rigid(case, seed)
    if kind == "relax_flex":
        return _relax_flexible(case, seed)
    if kind == "eval":
        m = _Flexible(case, seed)
        E, F, Ea = m.forces(flexible_start(case, seed)[0].double())
        return {"E": E, "F": F, "E_atom": Ea, "status": None}
    return _dynamics(case, seed)
