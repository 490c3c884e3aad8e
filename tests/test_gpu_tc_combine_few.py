"""Tensor-core combinations to few targets: tiles of 64 where 128 would not be resident.

Around the line (256 and 257 orbitals; 64 and 65 targets), past the orbitals whose coefficients
are resident in tiles of 64 (512 and 513), one target, point counts with and without a
remainder of 128; against FP64.

Tolerance: two BF16 slices hold an operand to 2^-17 and the dropped product of the low slices
is 2^-18 of the first, so every product is off by at most 2^-16 of its magnitude, whatever
the signs; FP32 sums of 600 terms add less.
"""
import ctypes as C
import subprocess

import pytest

from paper_1801_09263_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_orb", [256, 257, 288, 289, 299, 512, 513, 576, 577, 1030])
@pytest.mark.parametrize("n_targets", [1, 6, 63, 64, 65])
@pytest.mark.parametrize("points", [128 * 160, 128 * 153 + 4])
def test_few_targets_match_fp64(n_orb, n_targets, points):
    torch = pytest.importorskip("torch")
    lib = B.load_library()
    name = next(w for line in subprocess.run(["nm", "-D", B.library_path()], capture_output=True, text=True).stdout.splitlines()
                for w in line.split()[-1:] if w.startswith("_ZN4lace10tc_combineId"))
    fn = getattr(lib, name)
    P, I, S = C.c_void_p, C.c_int, C.c_size_t
    fn.argtypes = [I, S, I, P, S, P, I, C.c_double, P, S, P, P, P, P, P]
    gen = torch.Generator(device="cuda").manual_seed(n_orb + n_targets)
    a = torch.randn(n_orb, points, generator=gen, device="cuda")
    coef = torch.randn(n_orb, n_targets, generator=gen, dtype=torch.float64, device="cuda")
    out = torch.zeros(n_targets, points, dtype=torch.float64, device="cuda")
    scratch = torch.zeros(2 * 1280 * 256, dtype=torch.int32, device="cuda")
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    launches = C.c_int(0)
    assert fn(n_targets, points, n_orb, a.data_ptr(), points, coef.data_ptr(), n_targets, 0.0, out.data_ptr(), points,
              scratch.data_ptr(), flag.data_ptr(), None, None, C.addressof(launches)) == 0
    torch.cuda.synchronize()
    assert int(flag.item()) == 0
    a = a.double()
    bound = 2.0**-16 * (coef.abs().T @ a.abs())
    assert bool(((out - coef.T @ a).abs() <= bound).all())
