"""The context's wait limit bounds the grid barriers of the inverse square roots too.

With the limit at 0 a wait gives up at once, the CTAs leave the kernel by themselves and
the call returns LACE_ERR_TIMEOUT; with the default limit the same context gives what a
fresh one does.  More than 64 orbitals in mixed precision, more than 16 in FP64 (and in the FP64
alignment): the sizes that take a grid of CTAs.
"""
import numpy as np
import pytest

from paper_1801_09263_gb300 import LACE_FP64, LACE_MIXED, Lace, LaceError
from paper_1801_09263_gb300 import binding as B

pytestmark = pytest.mark.gpu

TIMEOUT, STATE = 6, 2
CELL, SHAPE = (7.0, 8.0, 9.0), (24, 24, 24)


def refused(call, *args):
    with pytest.raises(LaceError) as e:
        call(*args)
    return e.value.status


@pytest.mark.parametrize("prec,n", [(LACE_FP64, 24), (LACE_MIXED, 80)], ids=["fp64", "mixed"])
def test_short_limit_times_out_and_recovers(prec, n):
    phi = np.random.default_rng(n).standard_normal((n,) + SHAPE)
    with Lace(0, prec) as ref:
        ref.set_cell(CELL, SHAPE, 5.0)
        ref.load_orbitals(phi, n, 0, True)
        psi_ref = ref.get_orbitals(B.ORB_PSI)
        pivots = ref.localize(2)
        w_ref = ref.get_orbitals(B.ORB_PSI)
    with Lace(0, prec) as ctx:
        ctx.set_cell(CELL, SHAPE, 5.0)
        ctx.set_wait_limit(0.0)
        assert refused(ctx.load_orbitals, phi, n, 0, True) == TIMEOUT
        assert refused(ctx.get_orbitals, B.ORB_PSI) == STATE
        ctx.set_wait_limit(2.0)
        ctx.load_orbitals(phi, n, 0, True)
        assert np.array_equal(ctx.get_orbitals(B.ORB_PSI), psi_ref)
        ctx.set_wait_limit(0.0)
        assert refused(ctx.set_pivots, pivots) == TIMEOUT
        ctx.set_wait_limit(2.0)
        ctx.set_pivots(pivots)
        assert np.array_equal(ctx.get_orbitals(B.ORB_PSI), w_ref)
        assert ctx.align_to_previous() is False
        ctx.set_wait_limit(0.0)
        assert refused(ctx.align_to_previous) == TIMEOUT
        ctx.set_wait_limit(2.0)
        assert np.array_equal(ctx.get_orbitals(B.ORB_PSI), w_ref)
        assert ctx.align_to_previous() is True
