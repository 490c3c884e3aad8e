"""Exchanges of a few pairs, whose plane passes take wider CTAs, against the oracle.

One, two and five complex grids on cubes from the first size with wide CTAs (40) to the
last, so that launches lie on both sides of the line of one or two CTAs an SM.

Tolerance as for the lane passes at every other size: 3e-6 of the largest W, and
1e-6 Ha for E_x (up to ten pair energies of a few Ha with errors of ~1e-7).
"""
import numpy as np
import pytest

import oracle as O
import synth
from paper_1801_09263_gb300 import LACE_MIXED, Lace

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [36, 40, 48, 50, 54, 60, 64, 72, 80, 90, 96, 100, 108])
@pytest.mark.parametrize("n", [1, 2, 4])
def test_few_pairs_match_oracle(m, n):
    sysm = synth.small_localized_system(m + n, (10.0, 10.0, 10.0), (m, m, m), 8.0, n, n)
    g = O.Grid(sysm.cell, sysm.shape)
    occ = O.lowdin(g, sysm.phi)
    W_ref, ex_ref, _ = O.apply_exchange(g, occ, None, np.ones((n, n), dtype=bool))
    with Lace(0, LACE_MIXED) as ctx:
        ctx.set_cell(sysm.cell, sysm.shape, sysm.ecut)
        ctx.load_orbitals(sysm.phi, n, 0, True)
        W, ex = ctx.apply_exchange()
    assert abs(ex - ex_ref) <= 1e-6
    assert np.max(np.abs(W - W_ref)) <= 3e-6 * np.max(np.abs(W_ref))
