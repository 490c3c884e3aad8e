"""Loewdin orthonormalisation at the edges of its kernels' sizes, against the oracle.

Orbital counts at the tile edges of the FP64 Gram and combination (16), of the
inverse square root in one CTA (16, 32, 48, 64 rows in FP32, 16 in FP64) and by
a grid (tiles of 16 and 8 rows, 256 and 128 columns at a time), extras that make
the Gram rectangular, and a grid of an odd number of points.

Orbitals are noise, so the overlap's condition number is below 10.  Tolerances:
FP64 rounds sums of ~1e4 products (1e-16 each, random) and N x N products to below
1e-13 of the largest value, 1e-12 allowed; the mixed path's orbitals differ from the
symmetric Loewdin set by a rotation of ~1e-7 (FP32 Newton-Schulz) and FP32
rounding, 2e-6 of the largest value allowed, and are orthonormal to FP32's 24 bits.
"""
import numpy as np
import pytest

import oracle as O
from paper_1801_09263_gb300 import LACE_FP64, LACE_MIXED, Lace, LaceError
from paper_1801_09263_gb300 import binding as B

pytestmark = pytest.mark.gpu

CELL, SHAPE = (7.0, 8.0, 9.0), (27, 25, 25)


@pytest.mark.parametrize("prec,tol", [(LACE_FP64, 1e-12), (LACE_MIXED, 2e-6)], ids=["fp64", "mixed"])
@pytest.mark.parametrize("n_occ,n_extra", [(1, 0), (2, 1), (15, 3), (16, 0), (17, 5), (32, 0), (33, 16), (48, 17), (49, 0),
                                           (63, 1), (64, 0), (65, 0), (130, 20), (257, 0)])
def test_loewdin_sets_match_oracle(n_occ, n_extra, prec, tol):
    rng = np.random.default_rng(n_occ * 1000 + n_extra)
    phi = rng.standard_normal((n_occ + n_extra,) + SHAPE)
    g = O.Grid(CELL, SHAPE)
    ref = O.lowdin(g, phi[:n_occ])
    if n_extra:
        ref = np.concatenate([ref, O.orthonormalize_extras(g, ref, phi[n_occ:])])
    with Lace(0, prec) as ctx:
        ctx.set_cell(CELL, SHAPE, 5.0)
        ctx.load_orbitals(phi, n_occ, n_extra, True)
        psi = ctx.get_orbitals(B.ORB_PSI)
    assert np.max(np.abs(psi - ref)) <= tol * np.max(np.abs(ref))
    flat = psi.reshape(n_occ + n_extra, -1)
    s = g.dv * flat @ flat.T
    assert np.max(np.abs(s - np.eye(len(s)))) <= (1e-13 if prec == LACE_FP64 else 1e-6)


@pytest.mark.parametrize("prec", [LACE_FP64, LACE_MIXED], ids=["fp64", "mixed"])
@pytest.mark.parametrize("n", [4, 20, 40, 80])
def test_dependent_orbitals_are_refused(n, prec):
    phi = np.random.default_rng(n).standard_normal((n,) + SHAPE)
    phi[n - 1] = phi[0]
    with Lace(0, prec) as ctx:
        ctx.set_cell(CELL, SHAPE, 5.0)
        with pytest.raises(LaceError) as e:
            ctx.load_orbitals(phi, n, 0, True)
        assert e.value.status == 5
        phi[n - 1] = np.random.default_rng(1).standard_normal(SHAPE)
        ctx.load_orbitals(phi, n, 0, True)
