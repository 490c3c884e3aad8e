"""FP64 inverse square roots reach the rounding level, not only the stop test's bound.

The iteration is quadratic, so the residual of the step that passes the test lies anywhere
between the bound (1e-12 a diagonal element) and its square.  The matrices here have
the spectrum that just passes: eigenvalues 1 and a, with a such that the
scalar iteration x <- x (3 - x)^2 / 4 from x = lambda / ||A||_inf arrives at a sum of squares
of 0.8e-24 N.

Tolerance: X A X - I of a converged X is the rounding of a few products of N terms, 16 N
units of 1.1e-16 (4e-14 at 24 rows); what passes the test alone leaves 1e-12 here.
"""
import ctypes as C

import numpy as np
import pytest

from paper_1801_09263_gb300 import binding as B

pytestmark = pytest.mark.gpu


def residual(lam, c, steps):
    x = lam / c
    for _ in range(steps):
        x = x * (3.0 - x) ** 2 / 4.0
    return float(np.sum((1.0 - x) ** 2))


def just_passing(n, seed):
    """An orthogonal Q and a: Q diag(1 .. 1, a .. a) Q^T has residual 0.8e-24 n after some step."""
    q = np.linalg.qr(np.random.default_rng(seed).standard_normal((n, n)))[0]
    m = n // 2

    def at(a):
        lam = np.r_[np.ones(n - m), np.full(m, a)]
        mat = (q * lam) @ q.T
        mat = 0.5 * (mat + mat.T)
        return mat, lam, float(np.max(np.sum(np.abs(mat), axis=1)))

    _, lam, c = at(0.3)
    steps = next(k for k in range(60) if residual(lam, c, k) < 1e-26 * n)
    lo, hi = 1e-3, 0.3  # the residual falls with a
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        _, lam, c = at(mid)
        if residual(lam, c, steps) > 0.8e-24 * n:
            lo = mid
        else:
            hi = mid
    mat, lam, c = at(hi)
    assert 0.5e-24 * n < residual(lam, c, steps) < 1e-24 * n
    return mat


@pytest.mark.parametrize("n", [4, 16, 17, 24, 40, 130])
def test_fp64_inverse_sqrt_reaches_rounding(n):
    torch = pytest.importorskip("torch")
    fn = B.load_library()._ZN4lace12inv_sqrt_spdEiPKdPdS2_yPiP11CUstream_stS3_
    fn.argtypes = [C.c_int] + [C.c_void_p] * 3 + [C.c_ulonglong] + [C.c_void_p] * 3
    for seed in range(4):
        mat = just_passing(n, seed)
        a = torch.from_numpy(mat).cuda()
        x = torch.zeros_like(a)
        work = torch.zeros(5 * n * n + 320 * n + 320, dtype=torch.float64, device="cuda")
        status = torch.full((1,), -1, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        launches = C.c_int(0)
        assert fn(n, a.data_ptr(), x.data_ptr(), work.data_ptr(), 2 * 10**9, status.data_ptr(), None,
                  C.addressof(launches)) == 0
        torch.cuda.synchronize()
        assert int(status.item()) == 1
        x = x.cpu().numpy()
        assert np.max(np.abs(x @ mat @ x - np.eye(n))) <= 16 * n * 1.1e-16
