"""FP64 overlaps on both sides of the line between the 16- and the 64-wide tiles.

Square and rectangular overlaps whose 64-wide tiles are full or nearly so (256,
192 x 64, 128 x 128) and just past them (65, 257), on a point count that leaves a
remainder.  Orbitals are noise; sums of 1e4 products round at random: 1e-12 of the
largest value allowed, as for the other FP64 sets.
"""
import numpy as np
import pytest

import oracle as O
from paper_1801_09263_gb300 import LACE_FP64, Lace
from paper_1801_09263_gb300 import binding as B

pytestmark = pytest.mark.gpu

CELL, SHAPE = (7.0, 8.0, 9.0), (27, 25, 25)


@pytest.mark.parametrize("n_occ,n_extra", [(65, 64), (128, 128), (192, 64), (256, 0), (257, 2)])
def test_fp64_sets_match_oracle(n_occ, n_extra):
    phi = np.random.default_rng(n_occ).standard_normal((n_occ + n_extra,) + SHAPE)
    g = O.Grid(CELL, SHAPE)
    ref = O.lowdin(g, phi[:n_occ])
    if n_extra:
        ref = np.concatenate([ref, O.orthonormalize_extras(g, ref, phi[n_occ:])])
    with Lace(0, LACE_FP64) as ctx:
        ctx.set_cell(CELL, SHAPE, 5.0)
        ctx.load_orbitals(phi, n_occ, n_extra, True)
        psi = ctx.get_orbitals(B.ORB_PSI)
    assert np.max(np.abs(psi - ref)) <= 1e-12 * np.max(np.abs(ref))
