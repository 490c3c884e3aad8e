"""The rotation of the selected-column localisation on ill-conditioned column sets.

The square of the columns' condition number reaches 1e3 to 3e3 for noise at these
orbital counts.  The coupled Newton-Schulz iteration in FP32 leaves B^{-1/2} off by
delta ~ 6e-8 x that (2e-4), the first-order refinement makes it (3/4) delta^2 = 3e-8; the
localised orbitals are then orthonormal to that and FP32's rounding: 2e-7 allowed.  FP64:
delta ~ 1e-16 x 3e3, unrefined, 1e-11 allowed (sums over 400 orbitals).
"""
import numpy as np
import pytest

from paper_1801_09263_gb300 import LACE_FP64, LACE_MIXED, Lace
from paper_1801_09263_gb300 import binding as B

pytestmark = pytest.mark.gpu

CELL = (7.0, 8.0, 9.0)


@pytest.mark.parametrize("prec,tol", [(LACE_FP64, 1e-11), (LACE_MIXED, 2e-7)], ids=["fp64", "mixed"])
@pytest.mark.parametrize("n,shape", [(16, (12, 12, 12)), (17, (12, 12, 12)), (64, (20, 20, 20)), (65, (24, 24, 24)),
                                     (257, (36, 36, 36)), (400, (40, 40, 40))])
def test_localised_orbitals_stay_orthonormal(n, shape, prec, tol):
    phi = np.random.default_rng(n).standard_normal((n,) + shape)
    with Lace(0, prec) as ctx:
        ctx.set_cell(CELL, shape, 5.0)
        ctx.load_orbitals(phi, n, 0, True)
        ctx.localize(2)
        w = ctx.get_orbitals(B.ORB_PSI).reshape(n, -1)
    dv = np.prod(CELL) / w.shape[1]
    assert np.max(np.abs(dv * w @ w.T - np.eye(n))) <= tol
