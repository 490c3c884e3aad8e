"""FP32-accurate contractions on the tensor cores, against the oracle.

Orbital counts at the edges of the 128-wide tiles and of the 32-orbital steps, on
grids whose point counts leave a remainder in every tile (75 x 60 x 54 = 1898 x 128
+ 56, 54 x 50 x 45 = 949 x 128 + 28), with extras that make the overlap rectangular and
the projection accumulate; all above the size from which they replace the CUDA cores.

Tolerances.  The orbitals are noise: their overlap's condition number is below 2 and
their largest value 5 times the mean one.  Slices keep 2^-27 of a row's largest
value and results are rounded to FP32, both at random over > 1e5 points, so sums
are off by less than 1e-9; the inverse square root is refined to below 1e-10.  5e-8
of one is allowed for orthonormality (FP32 products reach 1.5e-7).  Orbitals differ
from the symmetric Loewdin set by FP32 rounding (6e-8) and a rotation of ~1e-7: 2e-6 of the
largest value.  Aligned sets span the same space, so they agree as well as two
rounded sets do: 1e-5 allowed.
"""
import numpy as np
import pytest

import oracle as O
from paper_1801_09263_gb300 import LACE_MIXED, Lace
from paper_1801_09263_gb300 import binding as B

pytestmark = pytest.mark.gpu

CELL = (7.0, 8.0, 9.0)


def overlap_error(g, psi):
    flat = psi.reshape(len(psi), -1)
    return np.max(np.abs(g.dv * flat @ flat.T - np.eye(len(flat))))


@pytest.mark.parametrize("shape,n_occ,n_extra", [((75, 60, 54), 65, 0), ((75, 60, 54), 96, 66), ((75, 60, 54), 127, 3),
                                                 ((75, 60, 54), 128, 0), ((54, 50, 45), 129, 96), ((54, 50, 45), 257, 0)])
def test_contractions_match_oracle(shape, n_occ, n_extra):
    rng = np.random.default_rng(n_occ)
    phi = rng.standard_normal((n_occ + n_extra,) + shape)
    g = O.Grid(CELL, shape)
    ref = O.lowdin(g, phi[:n_occ])
    if n_extra:
        ref = np.concatenate([ref, O.orthonormalize_extras(g, ref, phi[n_occ:])])
    with Lace(0, LACE_MIXED) as ctx:
        ctx.set_cell(CELL, shape, 5.0)
        ctx.load_orbitals(phi, n_occ, n_extra, True)
        psi = ctx.get_orbitals(B.ORB_PSI)
        assert np.max(np.abs(psi - ref)) <= 2e-6 * np.max(np.abs(ref))
        assert overlap_error(g, psi[:n_occ]) <= 5e-8
        # the rotation, and the alignment of another basis of the same space
        ctx.localize(2)
        assert ctx.align_to_previous() is False
        w = ctx.get_orbitals(B.ORB_PSI)[:n_occ]
        assert overlap_error(g, w) <= 1e-6
        turn = np.linalg.qr(rng.standard_normal((n_occ, n_occ)))[0]
        other = phi.copy()
        other[:n_occ] = (turn @ phi[:n_occ].reshape(n_occ, -1)).reshape((n_occ,) + shape)
        ctx.load_orbitals(other, n_occ, n_extra, True)
        ctx.localize(2)
        assert ctx.align_to_previous() is True
        w2 = ctx.get_orbitals(B.ORB_PSI)[:n_occ]
    assert np.max(np.abs(w2 - w)) <= 1e-5 * np.max(np.abs(w))


def test_rows_of_very_different_sizes():
    """Rows from 2^-40 to 2^40, already orthogonal: each is cut at its own scale."""
    shape, n = (75, 60, 54), 80
    g = O.Grid(CELL, shape)
    phi = O.lowdin(g, np.random.default_rng(5).standard_normal((n,) + shape))
    with Lace(0, LACE_MIXED) as ctx:
        ctx.set_cell(CELL, shape, 5.0)
        for e in (-40, 40):
            ctx.load_orbitals(phi * 2.0 ** e, n, 0, True)
            psi = ctx.get_orbitals(B.ORB_PSI)
            assert np.max(np.abs(psi - phi)) <= 2e-6 * np.max(np.abs(phi))
            assert overlap_error(g, psi) <= 5e-8
