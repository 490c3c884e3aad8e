"""One projector, one arithmetic: the kernels of an ACE build and apply depend on the
projector alone, not on how its functions come.

Small projectors run on the CUDA cores in FP32 (products and sums to ~2e-7 of the
largest value), larger ones on the tensor cores in split BF16 (~8e-6).  Sizes on both sides
of the line (3e6 values of 32^3 rows: 91 orbitals): host arrays, which are applied in four
chunks, device arrays, a part of a block alone, and the same system in a batch.  Between
routes only the grouping of FP32 partial sums may differ, 1e-6 of the largest value allowed;
batch and lone context (below the line) also accumulate W in another order.
"""
import numpy as np
import pytest

import synth
from paper_1801_09263_gb300 import LACE_MIXED, Lace
from paper_1801_09263_gb300 import binding as B

pytestmark = pytest.mark.gpu

TOL = 1e-6


def difference(a, b):
    return np.max(np.abs(a - b)) / np.max(np.abs(b))


@pytest.mark.parametrize("n,block", [(40, 100), (80, 100), (88, 150), (100, 30)])
def test_apply_takes_one_route(n, block):
    torch = pytest.importorskip("torch")
    sysm = synth.small_localized_system(n, (12.0, 12.0, 12.0), (32, 32, 32), 10.0, n, n)
    psi = np.random.default_rng(n).standard_normal((block,) + sysm.shape)
    with Lace(0, LACE_MIXED) as ctx:
        ctx.set_cell(sysm.cell, sysm.shape, sysm.ecut)
        ctx.load_orbitals(sysm.phi, n, 0, True)
        ctx.localize(2)
        ctx.screen(1e-3)
        ctx.apply_exchange()
        ctx.build_ace()
        host = ctx.apply_ace(psi)
        part = ctx.apply_ace(psi[:5])
        d_in = torch.from_numpy(psi).cuda()
        d_out = torch.empty_like(d_in)
        ctx.apply_ace_dev(d_in, d_out)
        dev = d_out.cpu().numpy()
    assert difference(host, dev) <= TOL
    assert difference(part, dev[:5]) <= TOL


def test_batch_builds_as_a_lone_context_does():
    systems = [synth.small_localized_system(s, (c, c, c), (m, m, m), 10.0, n, n)
               for s, c, m, n in ((1, 9.0, 24, 16), (2, 11.0, 32, 20))]
    with B.Batch([(s.cell, s.shape, s.ecut, s.n_occ, 1e-3) for s in systems]) as b:
        for q, s in enumerate(systems):
            b.set_orbitals(q, s.phi)
        for _ in range(3):  # eager, captured, replayed
            _, status = b.run()
            assert not status.any()
            xi = [b.context(q).get_orbitals(B.ORB_XI) for q in range(len(systems))]
    for s, x in zip(systems, xi):
        with Lace(0, LACE_MIXED) as ctx:
            ctx.set_cell(s.cell, s.shape, s.ecut)
            ctx.load_orbitals(s.phi, s.n_occ, 0, True)
            ctx.localize(2)
            ctx.screen(1e-3)
            ctx.apply_exchange()
            ctx.build_ace()
            lone = ctx.get_orbitals(B.ORB_XI)
        assert difference(x, lone) <= 4 * TOL
