"""Contexts in two threads whose calls need different amounts of dynamic shared
memory of the same kernels: neither call lowers the limit under the other's
launch."""
import threading
import time

import numpy as np
import pytest

from paper_2508_15522_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("what", ["eval", "relax", "rigid", "build"])
def test_calls_of_two_sizes_in_two_threads(what):
    import __graft_entry__ as ge
    ge.build()
    from paper_2508_15522_gb300 import gridff as G
    sub = synth.rocksalt_slab(ncell=1)
    box = synth.grid_box_for(sub, 0.5, height=6.0)
    errors, done = [], []
    until = time.monotonic() + 4.0

    def work(n, rcut):
        try:
            ctx = G.Context(0)
            if what == "rigid":
                grid = G.build_grid(ctx, sub, box.origin, box.length, box.spacing)
                mol = synth.rigid_molecule(n, 3)
                com, quat = synth.rigid_poses(mol, sub, 4, seed=1)
                x = np.concatenate([com, quat], 1).astype(np.float32).ravel()
            else:
                mol = synth.random_flexible_molecule(n, 3, 3)
                x = np.tile(mol.xyz.astype(np.float32).ravel(), 4)
            reps = G.Replicas(ctx, [mol], [0] * 4, rigid=what == "rigid")
            if what == "rigid":
                reps.set_launch_config(kernel=G.KERNEL_RIGID_SUBWARP, lanes_per_replica=32, warps_per_block=4,
                                       cache_slots=n)
            reps.set_state(x)
            while time.monotonic() < until and not errors:
                if what == "eval":
                    G.eval(ctx, None, reps, flags=G.NO_GRID)
                elif what == "relax":
                    G.relax(ctx, None, reps, 1, G.fire_params(f_conv=0.0), flags=G.NO_GRID)
                elif what == "rigid":
                    G.relax(ctx, grid, reps, 1, G.fire_params(f_conv=0.0))
                else:
                    G.build_grid(ctx, sub, box.origin, box.length, box.spacing, rcut=rcut).close()
                done.append(rcut)
            ctx.close()
        except Exception as e:          # noqa: BLE001  (reported below)
            errors.append((n, str(e)))

    # sizes that take the same kernel instance
    sizes = {"eval": ((9, 6.0), (120, 17.0)), "relax": ((17, 6.0), (32, 17.0)), "rigid": ((34, 6.0), (62, 17.0)),
             "build": ((9, 6.0), (9, 17.0))}[what]
    threads = [threading.Thread(target=work, args=s) for s in sizes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    assert len(set(done)) == 2
