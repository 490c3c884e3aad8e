"""A launch that fails is an error of the call, whichever of its launches it is.

A Gram is a kernel that sums chunks of the points and a second one that adds the
chunks; the small factorisations are chains of kernels.  Each runs here on a runtime
in which nothing runs and the k-th launch fails (fake_cudart.c), for every k: the call
has to return an error, and none without a failure (22 of the 25 failures were once
reported as success).  No GPU is needed.
"""
import os
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LIB = os.path.join(ROOT, "paper_1801_09263_gb300", "liblace.so")

PROGRAM = """
import ctypes as C, sys
lib = C.CDLL(sys.argv[1])
fake = C.CDLL(None)
P, I, S, D, Z = C.c_void_p, C.c_int, C.c_size_t, C.c_double, C.c_bool
n, at, launches = 1 << 12, 1 << 20, C.byref(C.c_int(0))  # nothing is read or written at these addresses
gemm = [I, I, S, P, S, P, S, D, Z, P, I, P, S, P, P], [40, 40, n, at, n, 2 * at, n, 1.0, False, at, 40, at, 1 << 22, None, launches]
calls = {
    "_ZN4lace9gemm_rowsIfEE9cudaErroriimPKT_mS4_mdbPdiS5_mP11CUstream_stPi": gemm,
    "_ZN4lace9gemm_rowsIdEE9cudaErroriimPKT_mS4_mdbPdiS5_mP11CUstream_stPi": gemm,
    "_ZN4lace10gram_exactEiimPKfPKjS1_S3_dPdiS4_mPiP11CUstream_stS5_": (
        [I, I, S, P, P, P, P, D, P, I, P, S, P, P, P], [40, 40, n, at, at, 2 * at, at, 1.0, at, 40, at, 1 << 22, at, None, launches]),
    "_ZN4lace7tc_gramEiimPKfmS1_mdPdiS2_mPiS3_P11CUstream_stS3_bb": (
        [I, I, S, P, S, P, S, D, P, I, P, S, P, P, P, P, Z, Z],
        [40, 40, n, at, n, 2 * at, n, 1.0, at, 40, at, 1 << 22, at, None, None, launches, False, False]),
    "_ZN4lace13lowdin_refineEiPdPKdS0_P11CUstream_stPi": ([I, P, P, P, P, P], [40, at, at, at, None, launches]),
    "_ZN4lace14cholesky_lowerEiPdiPiS1_P11CUstream_stS1_": ([I, P, I, P, P, P, P], [70, at, 70, at, None, None, launches]),
    "_ZN4lace11trtri_lowerEiPKdiPdiP11CUstream_stPi": ([I, P, I, P, I, P, P], [70, at, 70, at, 70, None, launches]),
}
for name, (types, args) in calls.items():
    fn = getattr(lib, name)
    fn.argtypes = types
    fake.fake_reset(0)
    ok = fn(*args)
    count = fake.fake_launched()
    bad = []
    for k in range(1, count + 1):
        fake.fake_reset(k)
        bad.append(fn(*args))
    print(name, ok, *bad)
"""


def test_failed_launches_are_reported(tmp_path):
    gcc = shutil.which("gcc")
    if not gcc or not os.path.exists(LIB):
        pytest.skip("needs gcc and the built liblace")
    so = tmp_path / "fake_cudart.so"
    r = subprocess.run([gcc, "-shared", "-fPIC", "-o", str(so), os.path.join(ROOT, "tests", "fake_cudart.c")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([sys.executable, "-c", PROGRAM, LIB], capture_output=True, text=True,
                         env=dict(os.environ, LD_PRELOAD=str(so), CUDA_VISIBLE_DEVICES="-1"))
    assert out.returncode == 0, out.stderr
    lines = out.stdout.strip().splitlines()
    assert len(lines) == 7
    for line in lines:
        name, ok, *bad = line.split()
        assert ok == "0" and len(bad) >= 2 and "0" not in bad, line
