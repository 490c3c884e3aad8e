"""The bytes that the request server admits a system by are those that it comes to hold.

After a whole step a context's buffers may exceed the prediction only by what it
leaves out, the axis tables and counters: below 32 KB at these sizes (5 axes' worth of
tables of at most 128 entries of 16 bytes, and lists of 12 bytes an orbital).  A grid on
the lane passes, an orthorhombic one, and an odd one on the generic passes.
"""
import ctypes as C

import numpy as np
import pytest

import synth
from paper_1801_09263_gb300 import LACE_FP64, LACE_MIXED, Lace
from paper_1801_09263_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [LACE_FP64, LACE_MIXED], ids=["fp64", "mixed"])
@pytest.mark.parametrize("shape,n,extra,block", [((64, 64, 64), 24, 0, 4), ((72, 80, 64), 40, 8, 16), ((45, 45, 45), 30, 0, 4)])
def test_prediction_covers_a_step(shape, n, extra, block, prec):
    fn = B.load_library()._ZN4lace17predict_ctx_bytesEiPKiiiim
    fn.restype = C.c_size_t
    fn.argtypes = [C.c_int, C.POINTER(C.c_int), C.c_int, C.c_int, C.c_int, C.c_size_t]
    sysm = synth.small_localized_system(1, tuple(0.3 * x for x in shape), shape, 6.0, n, n, extra)
    with Lace(0, prec) as ctx:
        ctx.set_cell(sysm.cell, shape, sysm.ecut)
        ctx.load_orbitals(sysm.phi, n, extra, True)
        ctx.localize(2)
        ctx.screen(1e-3)
        ctx.apply_exchange()
        ctx.build_ace()
        ctx.apply_ace(np.random.default_rng(0).standard_normal((block,) + shape))
        held = ctx.device_bytes()
    assert held - fn(prec, (C.c_int * 3)(*shape), n, extra, block, 2 << 30) <= 32 << 10
