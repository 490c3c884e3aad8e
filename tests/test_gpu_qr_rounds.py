"""SCDM pivoted QR in rounds (Sec. 2, FP32) at the edges of its phases.

Replaying the FP64 Gram-Schmidt steps of the oracle with the GPU's pivots,
every choice must be within 1e-4 of the largest residual norm (FP32 dots of up
to 520 products and squared norms downdated over the rounds: below 1e-5 of the
original norm, with residuals down to a tenth of it), and a second run must
pick the same pivots.  Cases: one pivot more and less than the 64 of a round; a
column count that is no multiple of four (4-byte copies); rows past 256 and 512
(one and two candidates a warp); a subsample of every point; and plane waves
in full shells, whose column norms are all the same, so that there are more
near-ties than candidates and a round takes the lowest index alone.
"""
import numpy as np
import pytest

import oracle as O
import synth
from paper_1801_09263_gb300 import LACE_MIXED, Lace, LaceError

pytestmark = pytest.mark.gpu


def check(cell, shape, ecut, phi, stride=2):
    n = len(phi)
    g = O.Grid(cell, shape)
    occ = O.lowdin(g, phi)
    with Lace(0, LACE_MIXED) as ctx:
        ctx.set_cell(cell, shape, ecut)
        ctx.load_orbitals(phi, n, 0, True)
        piv = ctx.localize(stride)
        assert np.array_equal(piv, ctx.localize(stride))
    assert len(set(piv.tolist())) == n
    sub = O.subsample_indices(g.shape, stride)
    pos = {int(v): k for k, v in enumerate(sub)}
    ratios = O.qrcp_pivot_ratios(occ.reshape(n, -1)[:, sub], [pos[int(p)] for p in piv])
    assert ratios.min() >= 1 - 1e-4, (ratios.min(), int(np.argmin(ratios)))


@pytest.mark.parametrize("shape,n,stride", [((32, 32, 32), 63, 2), ((32, 32, 32), 64, 2), ((32, 32, 32), 65, 2),
                                            ((45, 45, 45), 40, 2), ((27, 25, 30), 33, 2), ((36, 36, 36), 258, 2),
                                            ((40, 40, 40), 520, 2), ((24, 24, 24), 20, 1), ((24, 30, 32), 2, 3)],
                         ids=lambda v: str(v).replace(" ", ""))
def test_rounds_give_a_valid_qrcp_order(shape, n, stride):
    cell = (14.0, 14.0, 14.0)
    sysm = synth.small_localized_system(7 * n + shape[0], cell, shape, 10.0, max(2, (3 * n) // 4), n)
    check(cell, shape, 10.0, sysm.phi, stride)


def test_rounds_with_more_near_ties_than_candidates():
    # 1, cos and sin of every G of the first shell: each grid point has the density of any other
    n = 32
    x = 2.0 * np.pi * np.arange(n) / n
    one = np.ones((n, n, n))
    waves = [one]
    for a in range(3):
        ax = x.reshape([-1 if b == a else 1 for b in range(3)])
        waves += [np.cos(ax) * one, np.sin(ax) * one]
    check((10.0, 10.0, 10.0), (n, n, n), 20.0, np.array(waves))


def test_rounds_end_on_nan_orbitals():
    phi = synth.config1_plain().phi.copy()
    phi[3] = np.nan
    with Lace(0, LACE_MIXED) as ctx:
        ctx.set_cell((10.0, 10.0, 10.0), (24, 24, 24), 20.0)
        ctx.load_orbitals(phi, 8, 0, False)
        with pytest.raises(LaceError):
            ctx.localize(2)
