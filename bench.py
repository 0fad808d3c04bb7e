"""Benchmark of the GridFF hot path on GB300 (one JSON line on stdout).

Workload (the rigid-molecule configuration): a NaCl(001)-like slab
(a = 5.64 A, 8 x 8 primitive surface cells, 3 layers = 384 ions, +-0.7 e),
its 2a x 2a x 20 A tile on a 0.1 A grid (113 x 113 x 200 nodes, FP32
coefficients of the C, P, L channels), 4096 replicas of a planar 38-atom
C24H8O6 rigid core at random poses.  One step = one call relaxing every
replica for 2000 FIRE iterations from the initial poses with the force
threshold disabled, so that every replica does all iterations (the paper's
timing protocol, Sec. 6.4).  Inputs are seeded and synthetic.

Timing: W warm-up steps, then K steps, each bracketed by CUDA events on the
stream the library launches on; L2 is flushed (256 MB write) between steps,
outside the events.  value = atom-force evaluations per second (all ranks).
`e2e` times the same step through the public API with host buffers (pinned
pose upload, relaxation, pose/energy download) with a host clock.

--impl reference times the CPU oracle (the method's plain FP64 restatement)
on a bounded sample of the same workload on the host cores.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "atom-force evals/s"
UNIT = "atom-evals/s"
BYTES_PER_EVAL = 768          # 64 stencil nodes x 3 channels x 4 B (algorithmic)
N_REP = 4096
FIRE_ITERS = 2000
SEED = 1002
GHOST = 8                     # node planes below the grid floor (fit boundary far from the floor cells)


def workload():
    from paper_2508_15522_gb300 import synth
    sub = synth.rocksalt_slab(a=5.64, ncell=8, layers=3, charge=0.7)
    box = synth.grid_box_for(sub, 0.1, height=20.0)
    mol = synth.c24h8o6_core()
    com, quat = synth.rigid_poses(mol, sub, N_REP, seed=SEED)
    pose = np.concatenate([com, quat], 1).astype(np.float32)
    return sub, box, mol, pose


def config(extra=None):
    c = {"workload": "rigid C24H8O6 core x 4096 replicas, NaCl(001) 8x8x3 slab, 0.1 A grid "
                     "113x113x200 FP32 (C,P,L), 2000 FIRE iterations per step",
         "n_replicas": N_REP, "atoms_per_replica": 38, "fire_iterations_per_step": FIRE_ITERS,
         "grid": [113, 113, 200], "ghost_planes_below_floor": GHOST, "grid_bytes_fp32_padded": None,
         "l2_policy": "L2 flushed (256 MB write) between timed steps; the 44 MB grid is L2-resident "
                      "within a step by design"}
    if extra:
        c.update(extra)
    return c


# ---------------------------------------------------------------------------
# clocks during the timed region
# ---------------------------------------------------------------------------
class ClockSampler:
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device_index):
        self.dev = device_index
        self.rows = []          # (arrival time, fields)
        self.proc = None
        self.window = None      # (start, end) of the timed region

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.dev), f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "20"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
            t0 = time.perf_counter()     # sampling is running before the timed region starts
            while not self.rows and time.perf_counter() - t0 < 5.0 and self.proc.poll() is None:
                time.sleep(0.01)
        except (OSError, ValueError):
            self.proc = None
        return self

    def start(self):
        self.window = (time.perf_counter(), None)

    def stop(self):
        self.window = (self.window[0], time.perf_counter() + 0.05) if self.window else None

    def _read(self):
        for line in self.proc.stdout:
            parts = [p.strip() for p in line.split(",")]
            if len(parts) >= 9:
                self.rows.append((time.perf_counter(), parts))

    def __exit__(self, *a):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        rows = [r for t, r in self.rows if self.window and self.window[1] and self.window[0] <= t <= self.window[1]]
        if not rows:     # none arrived inside the window: the nearest ones around it
            rows = [r for _, r in self.rows[-3:]]
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"]}
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if "Active" in r[5 + i]
                          and "Not" not in r[5 + i]})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(rows)}


# ---------------------------------------------------------------------------
# CPU oracle (reported baseline / reference arm)
# ---------------------------------------------------------------------------
ORACLE_SAMPLE_REP = 128
ORACLE_SAMPLE_ITERS = 150        # cpu_baseline: ~10-30 s of CPU work
REFERENCE_STEP_ITERS = 40        # one --impl reference step: a few seconds


def oracle_sample(iters=ORACLE_SAMPLE_ITERS):
    """Rigid FIRE of the oracle on ORACLE_SAMPLE_REP replicas for
    ORACLE_SAMPLE_ITERS iterations on a coefficient grid of the full
    113 x 113 x 200 size (synthetic coefficients: only the cost is measured).
    Returns (atom-evals/s, seconds, sample description)."""
    from oracle import dynamics as odyn
    from oracle import grid as ogrid
    from paper_2508_15522_gb300 import synth
    sub, box, mol, pose = workload()
    n, h = ogrid.grid_dims(box.length, box.spacing)
    coefs = synth.random_coefficients(n, 3, seed=SEED, scale=(0.01, 0.01, 0.01))
    fn = odyn.make_force_fn(coefs, ("C", "P", "L"), box.origin, h, mol, intra=False)
    r = ORACLE_SAMPLE_REP
    t0 = time.perf_counter()
    odyn.fire_rigid(pose[:r, :3].astype(np.float64), pose[:r, 3:].astype(np.float64), np.zeros((r, 3)),
                    np.zeros((r, 3)), mol.xyz, mol.mass, fn, iters, odyn.FireParams(f_conv=0.0))
    dt = time.perf_counter() - t0
    evals = r * mol.n * iters
    desc = (f"{r} of the {N_REP} replicas x {iters} FIRE iterations on a full-size "
            f"113x113x200 coefficient grid (numpy FP64, single thread)")
    return evals / dt, dt, desc


def _oracle_worker(args):
    """One process of the all-cores oracle sample: rigid FIRE of replicas
    [lo, hi) (single-threaded numpy)."""
    lo, hi, iters = args
    from oracle import dynamics as odyn
    from oracle import grid as ogrid
    from paper_2508_15522_gb300 import synth
    sub, box, mol, pose = workload()
    n, h = ogrid.grid_dims(box.length, box.spacing)
    coefs = synth.random_coefficients(n, 3, seed=SEED, scale=(0.01, 0.01, 0.01))
    fn = odyn.make_force_fn(coefs, ("C", "P", "L"), box.origin, h, mol, intra=False)
    t0 = time.perf_counter()
    odyn.fire_rigid(pose[lo:hi, :3].astype(np.float64), pose[lo:hi, 3:].astype(np.float64), np.zeros((hi - lo, 3)),
                    np.zeros((hi - lo, 3)), mol.xyz, mol.mass, fn, iters, odyn.FireParams(f_conv=0.0))
    return (hi - lo) * mol.n * iters, time.perf_counter() - t0


def oracle_sample_all_cores(iters=ORACLE_SAMPLE_ITERS, per_proc=16):
    """The oracle sample spread over every host core: one spawned process per
    core, each relaxing `per_proc` replicas (numpy pinned to one thread per
    process).  Returns (atom-evals/s over the wall time of the parallel
    section, seconds, cores, description)."""
    import multiprocessing as mp
    cores = max(1, min(os.cpu_count() or 1, 64))
    for k in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS"):
        os.environ[k] = "1"
    jobs = [(k * per_proc, (k + 1) * per_proc, iters) for k in range(cores)]
    with mp.get_context("spawn").Pool(cores) as pool:
        pool.map(_oracle_worker, [(0, 1, 1)] * cores)          # start-up and imports, untimed
        t0 = time.perf_counter()
        res = pool.map(_oracle_worker, jobs)
        wall = time.perf_counter() - t0
    evals = sum(e for e, _ in res)
    desc = (f"{cores * per_proc} of the {N_REP} replicas x {iters} FIRE iterations on a full-size "
            f"113x113x200 coefficient grid (numpy FP64), {cores} processes x {per_proc} replicas, one per core")
    return evals / wall, wall, cores, desc


def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    for _ in range(args.warmup):
        pass   # the oracle has no warm-up state; warm-up steps are not timed
    vals = []
    for _ in range(args.steps):
        v, dt, cores, desc = oracle_sample_all_cores(REFERENCE_STEP_ITERS)
        vals.append((v, dt))
    value = statistics.mean(v for v, _ in vals)
    ms = statistics.mean(dt for _, dt in vals) * 1e3
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": config({"sample": desc}),
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": desc},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line))


# ---------------------------------------------------------------------------
# GPU arm
# ---------------------------------------------------------------------------
def kernel_source_hash():
    """Hash of the source the rigid sub-warp relaxation kernel is built
    from: the shared headers (internal.h, interp.cuh: cell location and
    B-spline weights, replica_common.cuh: record gathers), and of dynamics.cu
    the final-evaluation record and the sub-warp section (force routine,
    schedule, kernel).  Edits elsewhere in the file (flexible kernels, host
    code) leave the committed counters valid."""
    h = hashlib.sha256()
    csrc = os.path.join(ROOT, "paper_2508_15522_gb300", "csrc")
    for name in ("internal.h", "interp.cuh"):
        with open(os.path.join(csrc, name), "rb") as fh:
            h.update(fh.read())
    common = open(os.path.join(csrc, "replica_common.cuh"), encoding="utf-8").read()
    h.update(common.split("// 2^x by the PTX instruction")[0].encode())   # before the pair exponential
    src = open(os.path.join(csrc, "dynamics.cu"), encoding="utf-8").read()
    try:
        r0 = src.index("// Record of a replica's final evaluation")
        r1 = src.index("// Forces of one flexible replica whose positions are in s.x", r0)
        a = src.index("// FIRE, rigid replicas, sub-warp form")
        b = src.index("// FIRE, flexible replicas", a)
        h.update((src[r0:r1] + src[a:b]).encode())
    except ValueError:
        h.update(src.encode())
    return h.hexdigest()[:16]


def ncu_record():
    """The committed ncu figures of the relax kernel, if they were taken on
    the current kernel source (else {})."""
    p = os.path.join(ROOT, "profiles", "relax_rigid_c24h8o6_4096.json")
    try:
        d = json.load(open(p))
    except (OSError, ValueError):
        return {}
    return d if d.get("kernel_source_hash") == kernel_source_hash() else {}


def ncu_traffic():
    """DRAM bytes (read + write) per launch of the relax kernel from the
    committed ncu summary, if it was taken on the current kernel source
    (else None)."""
    return ncu_record().get("dram_bytes_per_launch")


def measured_peaks():
    try:
        return json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))
    except (OSError, ValueError):
        return {}


def reduce_over_ranks(seconds, evals, dist=None, device=None):
    """Whole-job figures of one timed region: (max seconds over ranks, sum of
    evaluations over ranks).  Replicas are independent, so this is the only
    cross-rank step (no data-path collective)."""
    if dist is None or not dist.is_initialized() or dist.get_world_size() == 1:
        return float(seconds), float(evals)
    import torch
    t = torch.tensor([float(seconds)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    e = torch.tensor([float(evals)], dtype=torch.float64, device=device)
    dist.all_reduce(e)
    return float(t.item()), float(e.item())


def mb_velocities(mol, n, seed):
    """(n, 6) rigid-body velocities (centre of mass, body angular) drawn
    from the 300 K Maxwell-Boltzmann distribution (synthetic NVE input)."""
    kT, acc = 0.025852, 9.648533e-3
    M = float(mol.mass.sum())
    b = mol.xyz
    I = np.array([np.sum(mol.mass * (np.sum(b * b, 1) - b[:, k] ** 2)) for k in range(3)])
    g = np.random.Generator(np.random.PCG64(seed + 7))
    return np.concatenate([g.standard_normal((n, 3)) * np.sqrt(kT * acc / M),
                           g.standard_normal((n, 3)) * np.sqrt(kT * acc / I)], 1).astype(np.float32)


def nve_drift(G, ctx, grid, reps, mol, pose, n_steps=10_000, dt=1.0, seed=SEED):
    """10k-step NVE (NO_SQUISH, 1 fs) of the relaxed replicas with 300 K
    Maxwell-Boltzmann velocities; returns the energy drift statistics and
    the NVE throughput (outside the timed region)."""
    n = len(pose)
    vel = mb_velocities(mol, n, seed)
    x, _ = reps.get_state()
    reps.set_state(x, vel.ravel())
    t0 = time.perf_counter()
    st, trace = G.run(ctx, grid, reps, n_steps, dt=dt, record_every=1000)
    wall = time.perf_counter() - t0
    d = np.abs(trace - trace[0:1])
    return {"steps": n_steps, "dt_fs": dt, "temperature_K": 300.0, "replicas": n,
            "max_abs_drift_eV": float(d.max()), "median_max_abs_drift_eV": float(np.median(d.max(0))),
            "atom_evals_per_s": n * mol.n * n_steps / (ctx.last_kernel_ms() * 1e-3),
            "wall_s": wall}


def minima_comparison(G, ctx, grid, mol, sub):
    """Minima found per second from learned proposals vs random starts.

    Training data: 64 batches of 16384 random-start relaxations (1.05 M;
    FIRE, |F| < 1e-3 eV/A, at most 2000 iterations).  Best-known set: the
    lowest converged energy among them; a hit is a converged relaxation
    within 0.01 eV of it.  The proposal network is trained (winner-takes-
    all, K = 8, 3000 Adam steps of 256 targets) on the hits.  Both arms then
    relax 4 batches of 16384 starts; the clock covers pose generation,
    relaxation and read-back of every batch."""
    from paper_2508_15522_gb300 import sampling as S
    a, n_rep = 5.64, 16384
    surf = S.Surface((0.0, 0.0), (a, a), sub.z_top + 3.0, sub.z_top + 5.0, sub.z_top + 2.0)
    sp = S.Sampler(ctx, grid, mol, surf, n_rep=n_rep, nsteps=FIRE_ITERS)
    E, P, T, C = [], [], [], []
    t0 = time.perf_counter()
    for k in range(64):
        b = sp.random_batch(10_000 + k)
        keep = b.converged
        E.append(b.energy[keep]); P.append(b.poses[keep]); T.append(sp.targets()[keep]); C.append(int(keep.sum()))
    gen_s = time.perf_counter() - t0
    E = np.concatenate(E)
    P = np.concatenate(P)
    T = np.concatenate(T)
    e_best = float(E.min())
    h = E <= e_best + 0.01
    best_set = len(sp.unique(P[h][:20000], E[h][:20000]))
    T = T[h]
    net = S.new_network(ctx, T, seed=1)
    t0 = time.perf_counter()
    losses = S.train_on_device(net, sp.desc, T, surf, 3000, batch=256, K=8, lr=1e-3, seed=7)
    train_s = time.perf_counter() - t0
    out = {"surface_tile_A": [a, a], "relaxations_for_training": 64 * n_rep, "converged_minima": int(sum(C)),
           "training_targets": int(h.sum()), "generation_s": gen_s, "best_known_eV": e_best,
           "best_known_unique": best_set, "tolerance_eV": 0.01, "rmsd_threshold_A": 0.1, "batches": 4,
           "replicas_per_batch": n_rep,
           "train": {"steps": 3000, "K": 8, "batch": 256, "seconds": train_s,
                     "loss_first": float(losses[:20].mean()), "loss_last": float(losses[-100:].mean())}}
    for name, fn in (("random", lambda k: sp.random_batch(20_000 + k)),
                     ("mlp", lambda k: sp.proposal_batch(net, 30_000 + k))):
        bs = [fn(k) for k in range(4)]
        wall = sum(b.wall_s for b in bs)
        hm = [S.hits(b, e_best) for b in bs]
        Ph = np.concatenate([b.poses[m] for b, m in zip(bs, hm)])
        Eh = np.concatenate([b.energy[m] for b, m in zip(bs, hm)])
        n_hits = int(sum(m.sum() for m in hm))
        out[name] = {"minima_per_s": n_hits / wall, "hits_per_s": n_hits / wall, "hits": n_hits,
                     "hit_fraction": n_hits / (4 * n_rep),
                     "converged_fraction": float(np.mean([b.converged.mean() for b in bs])),
                     "unique_of_best_set": len(sp.unique(Ph[:20000], Eh[:20000])) if n_hits else 0,
                     "wall_s": wall}
    out["gain"] = out["mlp"]["minima_per_s"] / max(out["random"]["minima_per_s"], 1e-30)
    out["amortised"] = amortised_gain(out, int(h.sum()), gen_s, train_s)
    net.close()
    sp.close()
    low = np.argsort(E, kind="stable")[:8]
    pr = G.Replicas(ctx, [mol], [0] * len(low), rigid=True)
    pr.set_state(np.ascontiguousarray(P[low], np.float32).ravel())
    xl = pr.positions().reshape(len(low), mol.n, 3)
    pr.close()
    out["error_vs_fp64_pairwise"] = grid_error_vs_pairwise(
        G, ctx, grid, sub, [(mol, v) for v in xl], "the 8 lowest converged minima of the training relaxations")
    return out


def amortised_gain(out, train_hits, gen_s, train_s):
    """The learned arm with the cost of its training: the random-start
    relaxations that found the training targets (gen_s, which found
    train_hits hits themselves) and the training (train_s) are charged to
    it, and their hits credited.  After N proposal batches of b hits in t
    seconds each: rate(N) = (train_hits + N b) / (gen_s + train_s + N t),
    gain(N) = rate(N) / random rate; break-even N where gain = 1."""
    r = out["random"]["hits_per_s"]
    b = out["mlp"]["hits"] / out["batches"]
    t = out["mlp"]["wall_s"] / out["batches"]
    res = {"training_data_s": gen_s, "training_s": train_s, "training_hits": train_hits,
           "proposal_batch_hits": b, "proposal_batch_s": t}
    for n in (out["batches"], 16, 64, 256):
        rate = (train_hits + n * b) / (gen_s + train_s + n * t)
        res[f"hits_per_s_after_{n}_batches"] = rate
        res[f"gain_after_{n}_batches"] = rate / max(r, 1e-30)
    den = b - r * t
    # None: the proposals never catch up; 0: ahead from the first batch (the
    # training relaxations found hits at least at the random-start rate)
    res["break_even_batches"] = max(0.0, (r * (gen_s + train_s) - train_hits) / den) if den > 0 else None
    return res


def flexible_minima_comparison(G, ctx):
    """The same comparison for a flexible molecule (24 atoms, 6 rotatable
    bonds): poses carry torsions and become positions through the pose
    builder.  Substrate: the NaCl(001) slab of the main workload with hard
    cations (synth.HARD_CATION, as the minima-hopping run), 0.1 A grid with
    8 ghost planes; on the soft-cation stand-in most proposals placed near
    the surface fall through the grid floor during relaxation (measured:
    82 % of them flagged below, 12 % accepted), which measures the
    stand-in's Pauli wall rather than the proposals.  Training data: 16
    batches of 8192 random-start relaxations (centre over the 5.64 A tile,
    uniform orientation and torsions); the network is trained (K = 8, 3000
    steps) on the poses of the converged minima within 0.05 eV of the
    best-known energy, or of the 256 lowest if that set is larger; hits are
    converged relaxations within 0.01 eV of it.  Both arms relax 16 batches
    of 8192 (hits are rare: about one per batch)."""
    from paper_2508_15522_gb300 import sampling as S
    from paper_2508_15522_gb300 import synth
    sub = synth.rocksalt_slab(a=5.64, ncell=8, layers=3, charge=0.7, cation_morse=synth.HARD_CATION)
    box = synth.grid_box_for(sub, 0.1, height=20.0)
    grid = G.build_grid(ctx, sub, box.origin, box.length, box.spacing, ghost_below=GHOST)
    a, n_rep, n_batch = 5.64, 8192, 16
    mol = synth.random_flexible_molecule(24, 6, 4242)
    surf = S.Surface((0.0, 0.0), (a, a), sub.z_top + 4.0, sub.z_top + 6.0, sub.z_top + 2.0)
    sp = S.FlexSampler(ctx, grid, mol, surf, n_rep=n_rep, nsteps=FIRE_ITERS)
    E, X, T, M = [], [], [], []
    t0 = time.perf_counter()
    for k in range(16):
        b = sp.random_batch(10_000 + k)
        Tk, Mk = sp.targets()
        keep = b.converged
        E.append(b.energy[keep]); X.append(b.poses[keep]); T.append(Tk[keep]); M.append(Mk[keep])
    gen_s = time.perf_counter() - t0
    E, X, T, M = (np.concatenate(v) for v in (E, X, T, M))
    e_best = float(E.min())
    # training set: every minimum within 0.05 eV of the best, at least the
    # 256 lowest (a handful of targets is learned poorly: measured, 95 targets
    # gave 5 hits in 4 proposal batches, the 288 within 0.1 eV gave 128)
    low = E <= max(e_best + 0.05, np.sort(E)[min(255, len(E) - 1)])
    h = E <= e_best + 0.01
    best_set = len(sp.unique(X[h], E[h]))
    net = S.new_network(ctx, T[low], seed=1)
    net.set_targets(T[low], M[low])
    t0 = time.perf_counter()
    losses = net.train(3000, 256, 8, sp.desc, 7, G.train_params(lr=1e-3, tile=surf.tile_xy))
    train_s = time.perf_counter() - t0
    out = {"atoms": mol.n, "rotatable_bonds": sp.n_rot, "relaxations_for_training": 16 * n_rep,
           "converged_minima": int(len(E)), "training_targets": int(low.sum()), "generation_s": gen_s,
           "best_known_eV": e_best, "best_known_hits": int(h.sum()), "best_known_unique": best_set,
           "tolerance_eV": 0.01, "batches": n_batch, "replicas_per_batch": n_rep,
           "substrate": "NaCl(001) 8x8x3 slab, charges +-0.7 e, hard cations (Morse R, eps of synth.HARD_CATION)",
           "train": {"steps": 3000, "K": 8, "batch": 256, "seconds": train_s,
                     "loss_first": float(losses[:20].mean()), "loss_last": float(losses[-100:].mean())}}
    for name, fn in (("random", lambda k: sp.random_batch(20_000 + k)),
                     ("mlp", lambda k: sp.proposal_batch(net, 30_000 + k))):
        bs = [fn(k) for k in range(n_batch)]
        wall = sum(b.wall_s for b in bs)
        hm = [S.hits(b, e_best) for b in bs]
        Xh = np.concatenate([b.poses[m] for b, m in zip(bs, hm)])
        Eh = np.concatenate([b.energy[m] for b, m in zip(bs, hm)])
        n_hits = int(sum(m.sum() for m in hm))
        out[name] = {"minima_per_s": n_hits / wall, "hits_per_s": n_hits / wall, "hits": n_hits,
                     "hit_fraction": n_hits / (n_batch * n_rep),
                     "converged_fraction": float(np.mean([b.converged.mean() for b in bs])),
                     "unique_hits": len(sp.unique(Xh[:20000], Eh[:20000])) if n_hits else 0, "wall_s": wall}
    out["gain"] = out["mlp"]["minima_per_s"] / max(out["random"]["minima_per_s"], 1e-30)
    out["amortised"] = amortised_gain(out, int(h.sum()), gen_s, train_s)
    net.close()
    sp.close()
    low = np.argsort(E, kind="stable")[:8]
    out["error_vs_fp64_pairwise"] = grid_error_vs_pairwise(
        G, ctx, grid, sub, [(mol, v) for v in X[low]],
        "the 8 lowest converged minima of the training relaxations (grid term)")
    grid.close()
    return out


def uneven_positions(G, reps, mols, tof, sub, seed):
    from paper_2508_15522_gb300 import synth
    x0 = np.zeros((reps.n_atoms, 3), np.float32)
    for k, m in enumerate(mols):
        idx = np.where(tof == k)[0]
        if len(idx) == 0:
            continue
        P = synth.flexible_positions(m, sub, len(idx), seed=seed + k)
        for j, r in enumerate(idx):
            x0[reps.atom_offset[r]:reps.atom_offset[r + 1]] = P[j]
    return x0.ravel()


def uneven_batch_comparison(G, ctx, grid, sub):
    """The batched persistent form against plain per-replica relaxation on
    16384 flexible replicas of 10-120 atoms (log-uniform, 0-12 torsion
    bonds, 256 generated templates), 1000 FIRE iterations per call.

    * batched: one persistent launch over all replicas with the autotuned
      layout, captured in a CUDA graph and replayed;
    * static: the same launch with the quad kernel and round-robin replica
      assignment (the layout before the tuner);
    * per-replica: one gridff_relax call per replica (a replica set of
      one), timed on 64 replicas of the batch (same starts) and scaled.
    Throughput runs use f_conv = 0 (every replica does every iteration).
    Minima runs use f_conv = 1e-3 eV/A; a relaxation is a minimum when it
    converged with finite values and no atom below the grid floor.
    Best-known energy per template: the lowest minimum of 8 further
    random-start batches of all 16384 replicas (batched form).  A hit is a
    minimum within 0.01 eV of its template's best-known energy; unique hits
    are the hits left after the RMSD-0.1 A filter per template.  hits/s and
    minima/s are per second of wall time of the arm's relaxation call."""
    from paper_2508_15522_gb300 import synth
    mols, tof = synth.uneven_batch(16384, 256, 77)
    reps = G.Replicas(ctx, mols, tof)
    x0 = uneven_positions(G, reps, mols, tof, sub, 5000)
    off = reps.atom_offset
    n_rep = len(tof)
    out = {"replicas": n_rep, "atoms": int(reps.n_atoms), "templates": len(mols), "fire_iterations": 1000,
           "f_conv_eV_per_A": 1e-3, "tolerance_eV": 0.01, "rmsd_threshold_A": 0.1}
    # trials as long as the calls they tune (1000 iterations): from random
    # starts the atoms change cell often in the first iterations, so short
    # trials understate the stencil caches against the long calls
    reps.set_state(x0)        # trials relax from the benchmark's starting structures
    best, log = G.tune(ctx, grid, reps, G.fire_params(f_conv=0.0), trial_steps=1000)
    out["tuned_config"] = best.as_dict()
    out["tuner_log"] = [[t["warps_per_block"], t["cache_slots"], t["queue"], t["l2_window"], t["cache_global"],
                         round(t["ms"], 2)] for t in log if t["kernel"] == G.KERNEL_FLEX_TERMS]
    out["tuner_log_fields"] = "unique-term kernel trials: warps per block, cache slots, queue, L2 window, global cache, ms"
    out["tuner_trials"] = len(log)

    def accepted_now():
        fs = reps.fire_state()
        x = reps.positions()
        lowest = np.minimum.reduceat(x[:, 2], off[:-1])
        ok = (((fs["status"] & G.REP_CONVERGED) != 0) & ((fs["status"] & G.REP_NONFINITE) == 0)
              & (lowest >= grid.floor))
        return ok, fs["energy"], x

    graphs = {}

    def batched(fconv):
        if fconv not in graphs:
            graphs[fconv] = G.RelaxGraph(ctx, grid, reps, 1000, G.fire_params(f_conv=fconv))
        return graphs[fconv].launch()

    # best-known energy of every template
    e_best = np.full(len(mols), np.inf)
    t0 = time.perf_counter()
    for k in range(8):
        reps.set_state(uneven_positions(G, reps, mols, tof, sub, 20_000 + 1000 * k))
        batched(1e-3)
        ok, E, _ = accepted_now()
        np.minimum.at(e_best, tof[ok], E[ok])
    out["best_known"] = {"batches": 8, "relaxations": 8 * n_rep, "seconds": time.perf_counter() - t0,
                         "templates_with_a_minimum": int(np.isfinite(e_best).sum())}

    def hits_of(ok, E, x, idx):
        """hits and unique hits among replicas idx (minima within tolerance)."""
        hit = ok & (E <= e_best[tof[idx]] + 0.01)
        uniq = 0
        for t in np.unique(tof[idx][hit]):
            sel = np.where(hit & (tof[idx] == t))[0]
            sel = sel[np.argsort(E[sel], kind="stable")]
            X = np.stack([x[off[idx[r]]:off[idx[r] + 1]] for r in sel])
            uniq += int((G.rmsd_unique_xyz(ctx, X, sub.tile, 0.1) < 0).sum())
        return int(hit.sum()), uniq

    def measure(label, runner):
        res = {}
        for fconv, key in ((0.0, "throughput"), (1e-3, "minima")):
            reps.set_state(x0)
            t0 = time.perf_counter()
            st, r = runner(fconv)
            wall = time.perf_counter() - t0
            ms = ctx.last_kernel_ms()
            if key == "throughput":
                res["atom_evals_per_s"] = r.atom_evals / (ms * 1e-3)
                res["replica_steps_per_s"] = n_rep * 1000 / (ms * 1e-3)
                res["kernel_ms"] = ms
            else:
                ok, E, x = accepted_now()
                n_hits, n_unique = hits_of(ok, E, x, np.arange(n_rep))
                res.update({"minima": int(ok.sum()), "minima_per_s": int(ok.sum()) / wall, "hits": n_hits,
                            "hits_per_s": n_hits / wall, "unique_hits": n_unique,
                            "unique_hits_per_s": n_unique / wall, "wall_s": wall})
        out[label] = res

    measure("batched", batched)
    for g in graphs.values():
        g.close()
    ok, _, xr = accepted_now()
    lowest = np.minimum.reduceat(xr[:, 2], off[:-1])
    out["batched"]["below_floor_after_relaxation"] = int((lowest < grid.floor).sum())
    pick = np.where(ok)[0]
    pick = pick[np.linspace(0, len(pick) - 1, 8).astype(int)] if len(pick) else pick
    out["error_vs_fp64_pairwise"] = grid_error_vs_pairwise(
        G, ctx, grid, sub, [(mols[tof[r]], xr[off[r]:off[r + 1]]) for r in pick],
        "8 minima (accepted relaxations) spread over the batch after the batched minima run (grid term)")
    reps.set_launch_config(G.LaunchConfig(kernel=G.KERNEL_FLEX_QUAD, lanes_per_replica=32, warps_per_block=4,
                                          cache_slots=48, queue=0, l2_window=0))
    measure("static", lambda fconv: G.relax(ctx, grid, reps, 1000, G.fire_params(f_conv=fconv)))
    reps.close()
    # plain per-replica relaxation of 64 replicas of the batch from the same starts
    sample = np.linspace(0, n_rep - 1, 64).astype(int)
    x0r = x0.reshape(-1, 3)
    wall, evals, ok_s, E_s, X_s = 0.0, 0, [], [], []
    for r in sample:
        m = mols[tof[r]]
        one = G.Replicas(ctx, [m], [0])
        one.set_state(np.ascontiguousarray(x0r[off[r]:off[r + 1]]).ravel())
        t0 = time.perf_counter()
        st, res = G.relax(ctx, grid, one, 1000, G.fire_params(f_conv=1e-3))
        wall += time.perf_counter() - t0
        evals += res.atom_evals
        fs = one.fire_state()
        xo = one.positions()
        ok_s.append(bool((fs["status"][0] & G.REP_CONVERGED) and not (fs["status"][0] & G.REP_NONFINITE)
                         and xo[:, 2].min() >= grid.floor))
        E_s.append(fs["energy"][0])
        X_s.append(xo)
        one.close()
    ok_s, E_s = np.array(ok_s), np.array(E_s)
    hit_s = ok_s & (E_s <= e_best[tof[sample]] + 0.01)
    per = wall / len(sample)
    out["per_replica"] = {"sampled_replicas": len(sample), "wall_s": wall, "projected_wall_s": per * n_rep,
                          "atom_evals_per_s": evals / wall, "minima": int(ok_s.sum()), "hits": int(hit_s.sum()),
                          "minima_per_s": int(ok_s.sum()) / wall, "hits_per_s": int(hit_s.sum()) / wall,
                          "hits_per_s_projected": out["batched"]["hits"] / (per * n_rep),
                          "projection": "the batched run's hits over the per-replica time of all 16384 relaxations "
                                        "(the same relaxations; the sampled hit count is small)"}
    bh = out["batched"]["hits_per_s"]
    out["hits_gain_vs_per_replica"] = bh / max(out["per_replica"]["hits_per_s_projected"], 1e-30)
    out["hits_gain_vs_static"] = bh / max(out["static"]["hits_per_s"], 1e-30)
    out["minima_gain_vs_per_replica"] = out["batched"]["minima_per_s"] / max(out["per_replica"]["minima_per_s"],
                                                                            1e-30)
    out["minima_gain_vs_static"] = out["batched"]["minima_per_s"] / max(out["static"]["minima_per_s"], 1e-30)
    return out


def precision_comparison(G, ctx):
    """Coefficient precision tiers on the neutral fcc(111) workload: a=4.08 A
    slab, 12 x 12 surface cells, 4 layers (576 atoms), Pauli and London
    channels only, 0.05 A grid over the 11.5 x 10.0 A tile and 20 A height;
    65536 rigid 24-atom molecules at random poses, 200 FIRE iterations per
    tier (f_conv = 0).  Error per tier: per-atom energy and force of 64
    replicas (1536 atoms) at their starting poses against the FP64 pairwise
    reference (direct Morse sums over the periodic slab)."""
    from oracle import substrate as osub
    from paper_2508_15522_gb300 import synth
    sub = synth.fcc111_slab(a=4.08, ncell=12, layers=4)
    box = synth.grid_box_for(sub, 0.05, height=20.0)
    mol = synth.rigid_molecule(24, 2024)
    n_rep = 65536
    com, quat = synth.rigid_poses(mol, sub, n_rep, seed=2025)
    pose = np.concatenate([com, quat], 1).astype(np.float32).ravel()
    sample = 64
    pts = None
    out = {"grid": None, "replicas": n_rep, "atoms_per_replica": mol.n, "fire_iterations": 200}
    errs = {}
    t0 = time.perf_counter()
    grid32 = G.build_grid(ctx, sub, box.origin, box.length, box.spacing, ghost_below=GHOST, channels=G.CH_P | G.CH_L,
                          keep_f64=True)
    out["build_s"] = time.perf_counter() - t0
    coefs = grid32.download_f64("coefs")
    out["grid"] = list(grid32.dims)
    for tier, st in (("f32", G.STORE_F32), ("f16", G.STORE_F16), ("bf16", G.STORE_BF16)):
        # every tier packs the same FP64 coefficients
        grid = grid32 if st == G.STORE_F32 else G.grid_from_coefs(ctx, coefs, grid32.origin, grid32.spacing,
                                                                  G.CH_P | G.CH_L, storage=st)
        reps = G.Replicas(ctx, [mol], [0] * n_rep, rigid=True)
        reps.set_state(pose)
        G.relax(ctx, grid, reps, 20, G.fire_params(f_conv=0.0))         # warm-up
        reps.set_state(pose)
        st_, res = G.relax(ctx, grid, reps, 200, G.fire_params(f_conv=0.0))
        ms = ctx.last_kernel_ms()
        # errors at the starting poses of the first `sample` replicas
        probe = G.Replicas(ctx, [mol], [0] * sample, rigid=True)
        probe.set_state(pose[:7 * sample])
        if pts is None:
            pts = probe.positions().astype(np.float64)
            Q = np.tile(mol.q, sample); R = np.tile(mol.R, sample); eps = np.tile(mol.eps, sample)
            E_ref, F_ref = osub.pairwise_reference(pts, Q, R, eps, sub)
        # per-atom grid energies and forces at those positions (flexible view)
        flex = G.Replicas(ctx, [mol], [0] * sample)
        flex.set_state(pts.astype(np.float32).ravel())
        E, F, Ea, S = G.eval(ctx, grid, flex, flags=G.NO_INTRA)
        errs[tier] = {"max_abs_dE_per_atom_eV": float(np.abs(Ea - E_ref).max()),
                      "rms_dE_per_atom_eV": float(np.sqrt(np.mean((Ea - E_ref) ** 2))),
                      "max_abs_dF_eV_per_A": float(np.abs(F - F_ref).max()),
                      "max_abs_dE_per_molecule_eV": float(np.abs(E - E_ref.reshape(sample, -1).sum(1)).max())}
        out[tier] = {"grid_bytes": grid.device_bytes, "kernel_ms": ms,
                     "atom_evals_per_s": res.atom_evals / (ms * 1e-3),
                     "replica_steps_per_s": n_rep * 200 / (ms * 1e-3), "error_vs_fp64_pairwise": errs[tier],
                     "scales": list(grid.scales)}
        for h in (flex, probe, reps):
            h.close()
        if grid is not grid32:
            grid.close()
    grid32.close()
    return out


def c2_accuracy(G, ctx, grid, sub, mol, pose, n_sample=8):
    """Error of the GPU energies and forces against the FP64 pairwise
    reference (direct Morse sums over the periodic slab and the EW3DC
    Ewald potential) for the first n_sample replicas at their start poses."""
    from oracle import dynamics as odyn
    from oracle import substrate as osub
    reps = G.Replicas(ctx, [mol], [0] * n_sample, rigid=True)
    reps.set_state(pose[:n_sample].ravel())
    E, F, Ea, S = G.eval(ctx, grid, reps)
    body = mol.xyz.astype(np.float32).astype(np.float64)
    x = odyn.rigid_positions(pose[:n_sample, :3].astype(np.float64), pose[:n_sample, 3:].astype(np.float64), body)
    t0 = time.perf_counter()
    Er, Fr = osub.pairwise_reference(x.reshape(-1, 3), np.tile(mol.q, n_sample), np.tile(mol.R, n_sample),
                                     np.tile(mol.eps, n_sample), sub)
    pair_s = time.perf_counter() - t0
    reps.close()
    return {"replicas": n_sample,
            "cpu_pairwise_fp64": {"value": n_sample * mol.n / pair_s, "unit": UNIT, "cores": 1,
                                  "sample": f"{n_sample} replicas x {mol.n} atoms, one evaluation each"},
            "max_abs_dE_per_molecule_eV": float(np.abs(E - Er.reshape(n_sample, -1).sum(1)).max()),
            "max_abs_dE_per_atom_eV": float(np.abs(Ea - Er).max()),
            "max_abs_dF_eV_per_A": float(np.abs(F - Fr).max()),
            "reference": "FP64 pairwise (Morse direct sums within 17 A + EW3DC Ewald)"}


def grid_error_vs_pairwise(G, ctx, grid, sub, items, what):
    """Error of the grid term at given molecule structures against the FP64
    pairwise reference of the substrate: `items` is a list of (molecule,
    positions (n, 3)); the GPU side is gridff_eval_points at those positions
    with the molecule's (Q, P, L) factors, the reference the oracle's direct
    Morse sums within 17 A plus the EW3DC Ewald potential.  Intramolecular
    terms are not part of either side."""
    from oracle import substrate as osub
    factors = {}
    x, qpl, q, R, eps, n_at = [], [], [], [], [], []
    for mol, xyz in items:
        if id(mol) not in factors:
            one = G.Replicas(ctx, [mol], [0])
            factors[id(mol)] = one.template_factors(0)
            one.close()
        x.append(np.asarray(xyz, np.float32).reshape(-1, 3))
        qpl.append(factors[id(mol)])
        q.append(mol.q); R.append(mol.R); eps.append(mol.eps); n_at.append(mol.n)
    x = np.concatenate(x)
    E, F, S = G.eval_points(ctx, grid, x, np.concatenate(qpl))
    t0 = time.perf_counter()
    Er, Fr = osub.pairwise_reference(x.astype(np.float64), np.concatenate(q), np.concatenate(R),
                                     np.concatenate(eps), sub)
    pair_s = time.perf_counter() - t0
    cut = np.cumsum([0] + n_at)
    dmol = [abs(float(E[a:b].astype(np.float64).sum() - Er[a:b].sum())) for a, b in zip(cut[:-1], cut[1:])]
    return {"structures": what, "molecules": len(items), "atoms": int(len(x)),
            "max_abs_dE_per_molecule_eV": max(dmol),
            "max_abs_dE_per_atom_eV": float(np.abs(E - Er).max()),
            "max_abs_dF_eV_per_A": float(np.abs(F - Fr).max()),
            "points_flagged": int(np.count_nonzero(S)), "pairwise_s": pair_s,
            "reference": "FP64 pairwise (Morse direct sums within 17 A + EW3DC Ewald)"}


def interpolation_roofline(G, ctx, grid, box, torch, dev, stream, l2_peak):
    """Grid interpolation alone (gridff_eval_points, no stencil reuse) at
    uniform random points over the tile and the z band [z0 + 2, z0 + 8] A:
    65536 x 38 = 2.49 M points per call with the grid factors of a 38-atom
    C/H/O set, 20 calls back to back on the stream (the grid stays
    L2-resident).  Two layouts: binned (the points put in cell order on the
    device by a counting sort, then one lane per point; the sort is inside
    the timed region) and direct (a quad of lanes per point in input
    order)."""
    from paper_2508_15522_gb300 import synth
    n_rep, n_at = 65536, 38
    g = synth.rng(3003)
    els = list(g.choice(["C", "H", "O"], n_at))
    R = np.array([synth.ELEMENTS[e][0] for e in els]); eps = np.array([synth.ELEMENTS[e][1] for e in els])
    pm = synth.Molecule(els, np.zeros((n_at, 3)), g.uniform(-0.3, 0.3, n_at), R, eps, np.full(n_at, 12.0))
    reps = G.Replicas(ctx, [pm], [0])
    qpl = np.tile(reps.template_factors(0), (n_rep, 1))
    reps.close()
    n = n_rep * n_at
    pts = synth.uniform_points(n, box, 3004, zband=(2.0, 8.0)).astype(np.float32)
    X = torch.from_numpy(pts.ravel()).to(dev)
    Q = torch.from_numpy(qpl.ravel()).to(dev)
    E = torch.empty(n, dtype=torch.float32, device=dev)
    F = torch.empty(3 * n, dtype=torch.float32, device=dev)
    out = {}
    for name, flags in (("binned", G.POINTS_BINNED), ("direct", 0)):
        for _ in range(3):
            G.eval_points(ctx, grid, X, Q, out=(E, F, None), flags=G.ASYNC | flags)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize(dev)
        e0.record(stream)
        iters = 20
        for _ in range(iters):
            G.eval_points(ctx, grid, X, Q, out=(E, F, None), flags=G.ASYNC | flags)
        e1.record(stream)
        torch.cuda.synchronize(dev)
        ms = e0.elapsed_time(e1) / iters
        achieved = BYTES_PER_EVAL * n / (ms * 1e-3) / 1e9
        out[name] = {"atom_evals_per_s": n / (ms * 1e-3), "ms_per_call": ms,
                     "roofline": {"bound": "l2", "achieved": achieved, "peak": l2_peak, "unit": "GB/s",
                                  "frac": achieved / l2_peak if l2_peak else None}}
    out["binned"]["kernels"] = ("bin_count_kernel, scan_tiles/scan_top/scan_apply_kernel, bin_scatter_kernel, "
                                "eval_sorted_kernel (lane per point); the sort is inside the timed region")
    out["direct"]["kernels"] = "eval_points_kernel (quad of lanes per point, input order)"
    best = max(("binned", "direct"), key=lambda k: out[k]["atom_evals_per_s"])   # the faster layout
    names = {"binned": "gridff_eval_points, binned layout (counting sort by cell + lane per point)",
             "direct": "gridff_eval_points, direct layout (quad of lanes per point, input order)"}
    return {"kernel": names[best], "layout": best,
            "atom_evals_per_s": out[best]["atom_evals_per_s"], "ms_per_call": out[best]["ms_per_call"],
            "points_per_call": n, "points": "uniform over the tile, z0 + [2, 8] A",
            "roofline": out[best]["roofline"], "layouts": out}


def minima_hopping_curve(G, ctx):
    """Minima hopping (Sec. 7) of a flexible 22-atom molecule on a NaCl(001)
    slab with a Cl vacancy (4 x 4 primitive cells, 3 layers, 95 atoms, hard
    cations: synth.hopping_substrate; grid over the 22.56 x 22.56 A defect
    period, 0.1 A, 8 ghost planes below the floor): 5000 replicas, 12 hops
    of 1000 Langevin steps at 300 K (dt 1 fs, gamma 0.01/fs), FIRE to
    1e-4 eV/A (at most 5000 iterations) and the RMSD-0.1 A filter against
    every minimum found so far; relaxed structures with an atom below the
    grid floor are no minima and restart from their initial structures.
    Returns the unique-minima-vs-time curve."""
    from paper_2508_15522_gb300 import sampling as S
    from paper_2508_15522_gb300 import synth
    sub = synth.hopping_substrate()
    box = synth.grid_box_for(sub, 0.1, height=20.0)
    t0 = time.perf_counter()
    grid = G.build_grid(ctx, sub, box.origin, box.length, box.spacing, ghost_below=GHOST)
    build_s = time.perf_counter() - t0
    mol = synth.random_flexible_molecule(22, 4, 2222)
    x0 = synth.flexible_positions(mol, sub, 5000, seed=2223, h_lo=3.5, h_hi=4.5, min_clear=3.0)
    mh = S.MinimaHopping(ctx, grid, mol, x0, sub.tile)
    curve = [mh.hop() for _ in range(12)]
    out = {"replicas": 5000, "atoms": mol.n, "grid": list(grid.dims), "grid_build_s": build_s, "hops": len(curve),
           "curve": [{"t_s": t, "unique_minima": u, "accepted": c, "restarted": b}
                     for (t, u, c), b in zip(curve, mh.below)],
           "lowest_eV": float(mh.db_E.min()) if len(mh.db_E) else None}
    if len(mh.db_E):
        low = np.argsort(mh.db_E, kind="stable")[:8]
        out["error_vs_fp64_pairwise"] = grid_error_vs_pairwise(
            G, ctx, grid, sub, [(mol, v) for v in mh.db_x[low]], "the 8 lowest unique minima found (grid term)")
    mh.close()
    grid.close()
    return out


def run_gpu(args):
    import torch
    import __graft_entry__ as ge
    ge.build()
    from paper_2508_15522_gb300 import gridff as G

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl" if torch.cuda.is_available() else "gloo")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    # one explicit stream for torch and the library: the legacy default
    # stream (handle 0) would make the context create its own stream, and
    # events recorded on the default stream would not bracket its kernels
    stream = torch.cuda.Stream(device=dev)
    torch.cuda.set_stream(stream)
    ctx = G.Context(local, stream=stream.cuda_stream)
    assert ctx.stream == stream.cuda_stream

    sub, box, mol, pose = workload()
    grid = G.build_grid(ctx, sub, box.origin, box.length, box.spacing, ghost_below=GHOST)
    reps = G.Replicas(ctx, [mol], [0] * N_REP, rigid=True)
    pose_dev = torch.from_numpy(pose.ravel()).to(dev)
    params = G.fire_params(f_conv=0.0)
    iters = args.fire_iters
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)

    def step():
        reps.set_state(pose_dev)
        st, res = G.relax(ctx, grid, reps, iters, params)
        return res

    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize(dev)
    if dist:
        dist.barrier()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    evals = 0
    kernel_ms = []
    with ClockSampler(local) as clk:
        torch.cuda.synchronize(dev)
        clk.start()
        for i in range(args.steps):
            flush.fill_(float(i))
            ev[i][0].record(stream)
            res = step()
            ev[i][1].record(stream)
            evals += res.atom_evals
            kernel_ms.append(ctx.last_kernel_ms())
        torch.cuda.synchronize(dev)
        clk.stop()
    step_ms = [a.elapsed_time(b) for a, b in ev]
    total_s, evals_all = reduce_over_ranks(sum(step_ms) / 1e3, evals, dist, dev)
    value = evals_all / total_s

    # end to end through the public API with host buffers (pinned)
    e2e_value = None
    if not args.quick:
        host_pose = torch.from_numpy(pose.ravel()).pin_memory()
        out_E = np.empty(N_REP, np.float64)
        e2e_s = []
        for i in range(max(1, min(args.steps, 5))):
            flush.fill_(float(i))
            torch.cuda.synchronize(dev)
            t0 = time.perf_counter()
            reps.set_state(host_pose.numpy())
            G.relax(ctx, grid, reps, iters, params)
            x, v = reps.get_state()
            out_E[:] = reps.fire_state()["energy"]
            e2e_s.append(time.perf_counter() - t0)
        e2e_value = N_REP * mol.n * iters / statistics.mean(e2e_s) * world

    # roofline of the dominant kernel (the fused relax kernel)
    l2_peak = hbm_read = None
    if not args.quick:
        l2_buf = torch.empty(48 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
        l2_peak = ctx.probe_read_bandwidth(l2_buf, iters=200)
        del l2_buf
        hbm_buf = torch.empty(2 * 1024 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
        hbm_read = ctx.probe_read_bandwidth(hbm_buf, iters=5)
        del hbm_buf
    k_ms = statistics.mean(kernel_ms)
    per_launch_evals = N_REP * mol.n * iters
    achieved = BYTES_PER_EVAL * per_launch_evals / (k_ms * 1e-3) / 1e9
    tpe = ncu_traffic()
    peaks = measured_peaks()
    clocks = clk.summary()
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": statistics.mean(step_ms), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": config({"grid_bytes_fp32_padded": grid.device_bytes, "parallelism": "replicas only",
                          "fire_iterations_per_step": iters}),
        "replica_steps_per_s": value / mol.n,
        "roofline": {"bound": "l2", "achieved": achieved, "peak": l2_peak, "unit": "GB/s",
                     "frac": (achieved / l2_peak) if l2_peak else None, "traffic": tpe,
                     "kernel": "relax_rigid_sw_kernel<W=16, R=3, F32x4>", "bytes_per_unit": BYTES_PER_EVAL,
                     "units_per_launch": per_launch_evals, "kernel_ms": k_ms,
                     "peak_source": "measured in this run: streaming read of a 48 MB L2-resident buffer "
                                    "(gridff_probe_read_bandwidth, best of 3 launch shapes)",
                     "hbm_peak_measured": peaks.get("hbm_gbs"), "hbm_read_this_run": hbm_read,
                     # measured context from the committed capture (None when the kernel changed since):
                     # the bytes actually read from L2 per eval and the SM issue activity
                     "l2_read_bytes_per_unit_measured": ncu_record().get("l2_to_l1_bytes_per_eval"),
                     "sm_issue_active_pct_measured": ncu_record().get("sm_issue_active_pct")},
        "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": 7 * 4 * N_REP,
                "d2h_bytes_per_step": (7 + 6) * 4 * N_REP + (5 * 4 + 8) * N_REP},
        "gpu_launches": 2 * args.steps,     # per step: fire_reset_kernel + the relaxation kernel
        "clocks": clocks,
    }
    if not args.quick:
        reps.set_state(pose_dev)
        G.relax(ctx, grid, reps, FIRE_ITERS, G.fire_params())
        line["nve_drift"] = nve_drift(G, ctx, grid, reps, mol, pose)
        line["minima"] = minima_comparison(G, ctx, grid, mol, sub)
        line["minima_flexible"] = flexible_minima_comparison(G, ctx)
        line["uneven_batch"] = uneven_batch_comparison(G, ctx, grid, sub)
        line["precision_tiers"] = precision_comparison(G, ctx)
        line["minima_hopping"] = minima_hopping_curve(G, ctx)
        line["interpolation_only"] = interpolation_roofline(G, ctx, grid, box, torch, dev, stream, l2_peak)
        line["accuracy_vs_fp64_pairwise"] = c2_accuracy(G, ctx, grid, sub, mol, pose)
    if rank == 0 and world == 1 and not args.quick:
        cv, cdt, ccores, cdesc = oracle_sample_all_cores()
        line["cpu_baseline"] = {"value": cv, "unit": UNIT, "cores": ccores, "kind": "oracle", "sample": cdesc}
        cv1, cdt1, cdesc1 = oracle_sample()
        line["cpu_baseline_1core"] = {"value": cv1, "unit": UNIT, "cores": 1, "kind": "oracle", "sample": cdesc1}
    if rank == 0:
        print(json.dumps(line))
    if dist:
        dist.barrier()
        dist.destroy_process_group()


def profile_case(args):
    """A small, self-contained launch of one kernel family for ncu captures
    (no JSON line): `uneven` relaxes 4096 of the uneven flexible replicas
    for 20 FIRE iterations; `langevin` runs 20 Langevin steps on them;
    `mlp` runs 20 training steps of the proposal network; `interp` evaluates
    the grid alone at 65536 x 38 uniform random points (gridff_eval_points,
    the interpolation-only workload of the bench line), twice in the direct
    layout, then twice binned; `nve` runs 200 rigid
    NVE steps of the bench's 4096 replicas, relaxed and given 300 K
    velocities as in the bench's NVE run; `fcc-f32`, `fcc-f16`, `fcc-bf16`
    relax the 65536 rigid replicas of the fcc(111) precision workload for 20
    FIRE iterations on the tier's grid.  Each runs its launch twice (the
    second is the one to capture with -s)."""
    import __graft_entry__ as ge
    ge.build()
    from paper_2508_15522_gb300 import gridff as G
    from paper_2508_15522_gb300 import synth
    ctx = G.Context(0)
    if args.profile_case in ("uneven", "langevin"):
        sub, box, _, _ = workload()
        grid = G.build_grid(ctx, sub, box.origin, box.length, box.spacing, ghost_below=GHOST)
        mols, tof = synth.uneven_batch(16384, 256, 77)
        tof = tof[:4096]
        reps = G.Replicas(ctx, mols, tof)
        x0 = uneven_positions(G, reps, mols, tof, sub, 5000)
        for _ in range(2):
            reps.set_state(x0)
            if args.profile_case == "uneven":
                G.relax(ctx, grid, reps, 20, G.fire_params(f_conv=0.0))
            else:
                G.langevin(ctx, grid, reps, 20, 1.0, 300.0, 0.01, 11)
        print(args.profile_case, "kernel ms", ctx.last_kernel_ms())
    elif args.profile_case == "mlp":
        from paper_2508_15522_gb300 import sampling as S
        g = np.random.default_rng(5)
        T = np.zeros((4096, G.MLP_OUT), np.float32)
        T[:, :3] = g.uniform(0, 5.64, (4096, 3))
        q = g.standard_normal((4096, 4))
        T[:, 3:7] = q / np.linalg.norm(q, axis=1, keepdims=True)
        net = S.new_network(ctx, T, seed=1)
        surf = S.Surface((0.0, 0.0), (5.64, 5.64), 0.0, 1.0, 0.0)
        for _ in range(2):
            S.train_on_device(net, np.zeros(S.N_DESC, np.float32), T, surf, 20, batch=256, K=8)
        print("mlp trained")
    elif args.profile_case == "nve":
        sub, box, mol, pose = workload()
        grid = G.build_grid(ctx, sub, box.origin, box.length, box.spacing, ghost_below=GHOST)
        reps = G.Replicas(ctx, [mol], [0] * N_REP, rigid=True)
        reps.set_state(pose.ravel())
        G.relax(ctx, grid, reps, FIRE_ITERS, G.fire_params(f_conv=0.0))      # as the bench's NVE run
        x, _ = reps.get_state()
        vel = mb_velocities(mol, N_REP, SEED)
        for _ in range(2):
            reps.set_state(x, vel.ravel())
            G.run(ctx, grid, reps, 200, dt=1.0)
        print("nve kernel ms", ctx.last_kernel_ms())
    elif args.profile_case in ("fcc-f32", "fcc-f16", "fcc-bf16"):
        sub = synth.fcc111_slab(a=4.08, ncell=12, layers=4)
        box = synth.grid_box_for(sub, 0.05, height=20.0)
        mol = synth.rigid_molecule(24, 2024)
        com, quat = synth.rigid_poses(mol, sub, 65536, seed=2025)
        pose = np.concatenate([com, quat], 1).astype(np.float32).ravel()
        grid32 = G.build_grid(ctx, sub, box.origin, box.length, box.spacing, ghost_below=GHOST,
                              channels=G.CH_P | G.CH_L, keep_f64=True)
        st = {"fcc-f32": G.STORE_F32, "fcc-f16": G.STORE_F16, "fcc-bf16": G.STORE_BF16}[args.profile_case]
        grid = grid32 if st == G.STORE_F32 else G.grid_from_coefs(ctx, grid32.download_f64("coefs"), grid32.origin,
                                                                  grid32.spacing, G.CH_P | G.CH_L, storage=st)
        reps = G.Replicas(ctx, [mol], [0] * 65536, rigid=True)
        for _ in range(2):
            reps.set_state(pose)
            G.relax(ctx, grid, reps, 20, G.fire_params(f_conv=0.0))
        print(args.profile_case, "kernel ms", ctx.last_kernel_ms(), "grid bytes", grid.device_bytes)
    elif args.profile_case == "interp":
        import torch
        sub, box, _, _ = workload()
        grid = G.build_grid(ctx, sub, box.origin, box.length, box.spacing, ghost_below=GHOST)
        n = 65536 * 38
        mol = synth.rigid_molecule(38, 3003)
        reps = G.Replicas(ctx, [mol], [0])
        qpl = np.tile(reps.template_factors(0), (65536, 1))
        pts = synth.uniform_points(n, box, 3004, zband=(2.0, 8.0)).astype(np.float32)
        dev = torch.device("cuda", 0)
        X = torch.from_numpy(pts.ravel()).to(dev)
        Q = torch.from_numpy(qpl.ravel()).to(dev)
        E = torch.empty(n, dtype=torch.float32, device=dev)
        F = torch.empty(3 * n, dtype=torch.float32, device=dev)
        for flags in (0, 0, G.POINTS_BINNED, G.POINTS_BINNED):
            G.eval_points(ctx, grid, X, Q, out=(E, F, None), flags=flags)
        print("interp evaluated (direct and binned)")


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="gridff", choices=["gridff", "reference"])
    ap.add_argument("--fire-iters", type=int, default=FIRE_ITERS,
                    help="FIRE iterations per step (profiling runs use a short step)")
    ap.add_argument("--quick", action="store_true",
                    help="skip the e2e leg, the bandwidth probes and the CPU baseline (profiling runs)")
    ap.add_argument("--profile-case", choices=["uneven", "langevin", "mlp", "interp", "nve", "fcc-f32", "fcc-f16",
                                               "fcc-bf16"], default=None,
                    help="run one small kernel case for an ncu capture and exit (no JSON line)")
    args = ap.parse_args()
    if args.profile_case:
        profile_case(args)
    elif args.impl == "reference":
        run_reference(args)
    else:
        run_gpu(args)


if __name__ == "__main__":
    main()
