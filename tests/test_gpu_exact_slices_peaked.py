"""The sliced contractions on peaked orbitals: what becomes of the tails.

Unmixed Gaussians of width 0.5 in a box of 20 on 96^3: the largest value of a row is
a hundred times its root mean square, and most points are far below 2^-6 of it, where a
row's fixed point (2^-30 of the largest value) has fewer bits than FP32.

Tolerances.  Orthonormality: the slices' error is at random over 8.8e5 points and adds
up to 1e-10; 5e-8 as for noise.  Pointwise: four units of 2^-30 of the largest value
(coefficients are close to the identity, sums over a few of them), plus FP32's share of the
orbitals that live there, the rotation of the inverse square root (1e-7) and the rounding
of inputs and results: 2e-6 of the largest value at the point.
"""
import numpy as np
import pytest

import oracle as O
from paper_1801_09263_gb300 import LACE_MIXED, Lace
from paper_1801_09263_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [72, 100])
def test_peaked_orbitals(n):
    m, edge, width = 96, 20.0, 0.5
    at = np.random.default_rng(n).uniform(0.0, edge, (n, 3))
    x = np.arange(m) * edge / m
    d = np.abs(x[None, None, :] - at[:, :, None])
    g1 = np.exp(-0.5 * (np.minimum(d, edge - d) / width) ** 2)
    phi = g1[:, 0, :, None, None] * g1[:, 1, None, :, None] * g1[:, 2, None, None, :]
    g = O.Grid((edge, edge, edge), (m, m, m))
    ref = O.lowdin(g, phi)
    assert np.max(np.abs(ref)) > 50.0 * np.sqrt(np.mean(ref**2))
    with Lace(0, LACE_MIXED) as ctx:
        ctx.set_cell((edge, edge, edge), (m, m, m), 5.0)
        ctx.load_orbitals(phi, n, 0, True)
        psi = ctx.get_orbitals(B.ORB_PSI)
    flat = psi.reshape(n, -1)
    assert np.max(np.abs(g.dv * flat @ flat.T - np.eye(n))) <= 5e-8
    peak = np.max(np.abs(ref))
    local = np.max(np.abs(ref), axis=0)
    assert np.mean(local < 2.0**-6 * peak) > 0.5
    assert (np.abs(psi - ref) <= 4.0 * 2.0**-30 * peak + 2e-6 * local).all()
