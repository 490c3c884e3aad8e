"""The tensor-core combination over orbitals at the edges of its variants.

Tiles of 128 targets (up to 128) and 256 (beyond), coefficients resident (up to
288 and 128 orbitals) or streamed, odd numbers of 32-orbital steps, and point
counts that leave a remainder (16 x 15 x 18 = 33 x 128 + 96) or not; against the same
application on the CUDA cores (LACE_NO_TC=1).

Tolerance: 3 x BF16 drops 2^-16 of a product of magnitudes and reads operands to
2^-17, at random signs over up to 300 orbitals and two contractions: 1e-4 of the
largest value allowed.
"""
import numpy as np
import pytest

from paper_1801_09263_gb300 import LACE_MIXED, Lace

pytestmark = pytest.mark.gpu

CELL = (7.0, 8.0, 9.0)


@pytest.mark.parametrize("n_occ,n_apply,shape", [(1, 1, (16, 15, 18)), (70, 129, (16, 15, 18)), (65, 128, (16, 16, 16)),
                                                 (128, 190, (16, 15, 18)), (129, 190, (16, 15, 18)), (300, 3, (20, 18, 16)),
                                                 (290, 300, (16, 15, 18))])
def test_apply_matches_cuda_cores(n_occ, n_apply, shape, monkeypatch):
    rng = np.random.default_rng(n_occ + n_apply)
    phi = rng.standard_normal((n_occ,) + shape)
    psi = rng.standard_normal((n_apply,) + shape)
    out = []
    with Lace(0, LACE_MIXED) as ctx:
        ctx.set_cell(CELL, shape, 5.0)
        ctx.load_orbitals(phi, n_occ, 0, True)
        ctx.apply_exchange(False)
        ctx.build_ace()
        for off in ("0", "1"):
            monkeypatch.setenv("LACE_NO_TC", off)
            out.append(ctx.apply_ace(psi))
    assert np.max(np.abs(out[0] - out[1])) <= 1e-4 * np.max(np.abs(out[1]))
