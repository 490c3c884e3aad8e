"""The lane passes of the pair convolutions on boxes and cubes, against the oracle.

Sizes at the edges of what the passes accept and of their index arithmetic:
24 and 128 points an axis, odd x and y axes, every radix pair of the x and y
axes and of half the z axis, rows of 4k + 2 points (8-byte orbital reads and W
updates), column counts that leave the last slab of pass B partly empty, and a
grid whose last complex grid holds one pair.

Tolerance: two transforms of at most six radix stages, each rounding to about
one unit (6e-8) of the running magnitude a stage, add up to below 5e-7 rms of
the largest W; the largest of ~1e6 errors is within six times that: 3e-6.
E_x sums at most six pair energies of a few Ha with errors of ~1e-7: 1e-6.
"""
import numpy as np
import pytest

import oracle as O
import synth
from paper_1801_09263_gb300 import LACE_MIXED, Lace

pytestmark = pytest.mark.gpu

SHAPES = [(24, 24, 24), (25, 27, 30), (27, 25, 54), (45, 75, 50), (75, 45, 90), (81, 32, 36), (24, 128, 24),
          (128, 24, 32), (24, 24, 128), (30, 36, 40), (40, 48, 60), (54, 50, 64), (60, 64, 72), (72, 80, 64),
          (90, 30, 48), (100, 96, 80), (108, 120, 25 * 4), (120, 40, 108), (32, 54, 120), (64, 90, 96), (96, 81, 24),
          (80, 100, 30), (48, 108, 48), (36, 60, 128), (108, 108, 108), (120, 120, 120), (90, 90, 90), (30, 30, 30)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_lane_passes_match_oracle(shape):
    # the spacing of the grids differs per axis: cells of 8-16 bohr, 3 orbitals (2 full grids and 1 half)
    cell = tuple(8.0 + 8.0 * n / 128.0 for n in shape)
    sysm = synth.small_localized_system(sum(shape), cell, shape, 8.0, 2, 2, 1)
    g = O.Grid(sysm.cell, sysm.shape)
    occ = O.lowdin(g, sysm.phi[:2])
    extra = O.orthonormalize_extras(g, occ, sysm.phi[2:])
    W_ref, ex_ref, _ = O.apply_exchange(g, occ, extra, np.ones((2, 3), dtype=bool))
    with Lace(0, LACE_MIXED) as ctx:
        ctx.set_cell(sysm.cell, sysm.shape, sysm.ecut)
        ctx.load_orbitals(sysm.phi, 2, 1, True)
        W, ex = ctx.apply_exchange()
        pairs = ctx.get_pairs()
    assert len(pairs) == 5
    assert abs(ex - ex_ref) <= 1e-6
    assert np.max(np.abs(W - W_ref)) <= 3e-6 * np.max(np.abs(W_ref))
