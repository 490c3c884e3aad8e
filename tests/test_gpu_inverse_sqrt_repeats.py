"""Inverse square roots by a grid of CTAs give the same bits every time.

All sums of the load run in a fixed order, so a part of the result that a CTA
did not write, or a step too many, shows as a difference.  Orbital counts of a few tiles (8
rows in FP64, 16 in FP32) up to more tiles than CTAs; noise on a small grid, so that most
of a load is the iteration.
"""
import numpy as np
import pytest

from paper_1801_09263_gb300 import LACE_FP64, LACE_MIXED, Lace
from paper_1801_09263_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n", [(LACE_FP64, 17), (LACE_FP64, 40), (LACE_FP64, 160), (LACE_MIXED, 65), (LACE_MIXED, 300)])
def test_repeated_loads_are_identical(prec, n):
    shape = (12, 12, 12)
    phi = np.random.default_rng(n).standard_normal((n,) + shape)
    with Lace(0, prec) as ctx:
        ctx.set_cell((5.0, 5.0, 5.0), shape, 5.0)
        ctx.load_orbitals(phi, n, 0, True)
        first = ctx.get_orbitals(B.ORB_PSI)
        for _ in range(100):
            ctx.load_orbitals(phi, n, 0, True)
            assert np.array_equal(ctx.get_orbitals(B.ORB_PSI), first)
