"""Node values of gridff_build_grid against the oracle's direct sums, at the
sizes and parameters where the tabulated radial functions, the item edges
(4 columns, 32 planes) and the selection of reciprocal vectors can go wrong.

Tolerances (derived before the first run).  Morse channels: every term is
positive and its relative error is that of an FP64 exponential of an argument
up to alpha d = 35 (8e-15), so a node's sum is held to 1e-12 of itself.  The
cutoffs are chosen so that no lattice distance falls on them.  Coulomb
channel: both sides use the same Ewald parameters; the vectors left out have
structure factors below 2^-46 of the sum of |q|, at most 4e-12 V together,
and the sums round at 1e-13: held to 1e-10 of the largest value.
"""
import numpy as np
import pytest

from oracle import grid as ogrid
from oracle import substrate as osub
from paper_2508_15522_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import __graft_entry__ as ge
    ge.build()
    from paper_2508_15522_gb300 import gridff
    return gridff, gridff.Context(0)


SLABS = {
    "rocksalt": lambda: synth.rocksalt_slab(ncell=2, layers=2),
    "vacancy": lambda: synth.with_top_vacancy(synth.rocksalt_slab(ncell=2, layers=2)),
    "metal": lambda: synth.fcc111_slab(ncell=4, layers=2),
}


@pytest.mark.parametrize("slab, spacing, height, gap, alpha, rcut", [
    ("rocksalt", 0.71, 4.3, 1.0, 1.5, 16.937),     # fewer planes than an item, ragged columns
    ("rocksalt", 0.62, 20.0, 1.0, 1.5, 16.937),    # more than one item along z, planes beyond the cutoff
    ("rocksalt", 0.83, 3.9, 0.23, 1.5, 9.613),     # nodes closer than 0.5 A to atoms (no table there)
    ("rocksalt", 0.77, 5.1, 1.0, 2.5, 14.137),     # alpha rcut > 30: the functions called directly
    ("rocksalt", 0.77, 5.1, 1.0, 2.1, 14.137),     # the steepest exponent the table takes
    ("vacancy", 0.93, 5.3, 1.0, 1.5, 11.937),      # every reciprocal vector kept
    ("metal", 0.69, 6.1, 1.0, 1.5, 12.413),        # Morse channels only
])
def test_node_values_match_direct_sums(env, slab, spacing, height, gap, alpha, rcut):
    G, ctx = env
    sub = SLABS[slab]()
    origin = (0.13, -0.21, sub.z_top + gap)
    length = (sub.tile[0], sub.tile[1], height)
    grid = G.build_grid(ctx, sub, origin, length, spacing, alpha=alpha, rcut=rcut, keep_f64=True)
    channels = ("C", "P", "L") if np.any(sub.q) else ("P", "L")
    ref, n, _ = ogrid.node_values(sub, origin, length, spacing, channels, alpha, rcut,
                                  osub.ewald_params(1e-10, 12.0) if "C" in channels else None)
    got = grid.download_f64("values")
    assert got.shape == ref.shape == (len(channels),) + n
    for c, ch in enumerate(channels):
        err = np.abs(got[c] - ref[c])
        if ch == "C":
            assert err.max() <= 1e-10 * np.abs(ref[c]).max(), (ch, err.max())
        else:
            assert (err <= 1e-12 * np.abs(ref[c])).all(), (ch, (err / np.maximum(np.abs(ref[c]), 1e-300)).max())
