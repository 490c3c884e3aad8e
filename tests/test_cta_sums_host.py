"""Sums over the CTAs of a persistent kernel: no part is overwritten before it is read.

The inverse square roots by a grid sum their convergence measure and, right after the
last test, a norm over the CTAs; a CTA late by a few hundred nanoseconds must still
find the parts of the sum that it is at.  A host model of the schedule, built from
the header that the kernel uses, holds each CTA back in turn.  No GPU is needed.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1801_09263_gb300", "csrc")


def test_parts_outlive_their_readers(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = tmp_path / "cta_sums_check"
    r = subprocess.run([nvcc, "-std=c++17", "-I", CSRC, os.path.join(ROOT, "tests", "cta_sums_check.cu"), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout
