"""The order of the kept pairs of localised orbitals, made on the device.

Rows and columns of the list run through the orbitals along the Z-order curve of
their grid points (coordinate bits interleaved, the first axis highest), the
pairs with the extras at the end of each row; every pair has its lower orbital
first.  Exact comparison with the definition, at orbital counts around the
blocks of 256 and with pivots found by the factorisation or imposed.
"""
import numpy as np
import pytest

from paper_1801_09263_gb300 import LACE_MIXED, Lace
from paper_1801_09263_gb300 import binding as B

pytestmark = pytest.mark.gpu

CELL = (7.0, 8.0, 9.0)


def z_code(p, shape):
    x, y, z = np.unravel_index(int(p), shape)
    return sum((int(x) >> b & 1) << 3 * b + 2 | (int(y) >> b & 1) << 3 * b + 1 | (int(z) >> b & 1) << 3 * b for b in range(8))


@pytest.mark.parametrize("n_occ,n_extra,shape,thr", [(1, 0, (8, 10, 12), 0.0), (2, 3, (8, 10, 12), 0.0), (40, 2, (12, 15, 16), 0.02),
                                                     (257, 1, (20, 18, 16), 0.6)])
def test_pairs_follow_the_z_order(n_occ, n_extra, shape, thr):
    rng = np.random.default_rng(n_occ)
    phi = rng.standard_normal((n_occ + n_extra,) + shape)
    with Lace(0, LACE_MIXED) as ctx:
        ctx.set_cell(CELL, shape, 5.0)
        ctx.load_orbitals(phi, n_occ, n_extra, True)
        piv = np.array(ctx.localize(2))
        for imposed in (False, True):
            if imposed:
                piv = piv[rng.permutation(n_occ)]
                ctx.set_pivots(piv)
            n_pairs = ctx.screen(thr)
            got = np.array(ctx.get_pairs()).reshape(-1, 2)
            s = ctx.get_matrix(B.MAT_OVERLAP_MODULI)
            order = sorted(range(n_occ), key=lambda i: (z_code(piv[i], shape), i))
            want = []
            for r, i in enumerate(order):
                row = [(min(i, j), max(i, j)) for j in order[r:]]
                want += [p for p in row if s[p] >= thr] + [(i, n_occ + e) for e in range(n_extra)]
            assert n_pairs == len(want)
            assert np.array_equal(got, np.array(want))
