"""A refused inverse square root leaves its output as it was, whichever kernel ran.

A diagonal matrix of condition 1e13 converges exactly and is refused by the limit on
the condition number (1e12); a singular one does not converge.  Rows: one CTA (up to 16), a
cluster (17 to 64 in FP32), a grid.
"""
import ctypes as C

import numpy as np
import pytest

from paper_1801_09263_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["_ZN4lace12inv_sqrt_spdEiPKdPdS2_yPiP11CUstream_stS3_",
                                  "_ZN4lace18inv_sqrt_spd_mixedEiPKdPdS2_yPiP11CUstream_stS3_"], ids=["fp64", "fp32"])
@pytest.mark.parametrize("n", [12, 30, 60, 100])
@pytest.mark.parametrize("last", [1e-13, 0.0, 1e-3])
def test_output_is_written_only_on_success(name, n, last):
    torch = pytest.importorskip("torch")
    fn = getattr(B.load_library(), name)
    fn.argtypes = [C.c_int] + [C.c_void_p] * 3 + [C.c_ulonglong] + [C.c_void_p] * 3
    diag = np.ones(n)
    diag[-1] = last
    a = torch.from_numpy(np.diag(diag)).cuda()
    x = torch.full_like(a, 7.0)
    work = torch.zeros(5 * n * n + 320 * n + 320, dtype=torch.float64, device="cuda")
    status = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    launches = C.c_int(0)
    assert fn(n, a.data_ptr(), x.data_ptr(), work.data_ptr(), 2 * 10**9, status.data_ptr(), None,
              C.addressof(launches)) == 0
    torch.cuda.synchronize()
    if last == 1e-3:
        assert int(status.item()) == 1
        assert np.allclose(x.cpu().numpy(), np.diag(diag ** -0.5), rtol=1e-5, atol=1e-6)
    else:
        assert int(status.item()) == 0
        assert bool((x == 7.0).all())
