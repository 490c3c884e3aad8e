"""A value that is not a number spoils its own grid point, not its orbital.

The rotation of unnormalised orbitals with imposed points, at a size that takes the sliced
tensor-core kernels, with a NaN in one orbital and an infinity in another: away from
these two points the result has the bits of the rotation without them, for
orbitals small, ordinary and beyond the range of the slices' FP16.
"""
import numpy as np
import pytest

from paper_1801_09263_gb300 import LACE_MIXED, Lace
from paper_1801_09263_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [1e-4, 1.0, 1e6])
def test_nonfinite_values_stay_at_their_points(size):
    n, shape = 80, (75, 60, 54)
    phi = size * np.random.default_rng(7).standard_normal((n,) + shape)
    with Lace(0, LACE_MIXED) as ctx:
        ctx.set_cell((7.0, 8.0, 9.0), shape, 5.0)
        ctx.load_orbitals(phi, n, 0, False)
        pivots = ctx.localize(2)
        clean = ctx.get_orbitals(B.ORB_PSI).reshape(n, -1)
        # two points that are neither pivots nor the largest values of their rows
        free = [p for p in (12345, 200000, 54321, 99999) if p not in pivots]
        for row, point, value in ((3, free[0], np.nan), (41, free[1], np.inf)):
            assert abs(phi[row].flat[point]) < np.max(np.abs(phi[row]))
            phi[row].flat[point] = value
        ctx.load_orbitals(phi, n, 0, False)
        ctx.set_pivots(pivots)
        w = ctx.get_orbitals(B.ORB_PSI).reshape(n, -1)
    assert not np.isfinite(w[:, free[:2]]).any()
    rest = np.ones(w.shape[1], dtype=bool)
    rest[free[:2]] = False
    assert np.array_equal(w[:, rest], clean[:, rest])
