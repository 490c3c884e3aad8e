"""REBUILDs of one group are announced to the executor before any of them runs (CPU only).

The merged pair convolutions wait for the REBUILDs that they know of.  When each
announced itself as its thread started, one that started a millisecond late was not waited
for, and rebuilds take little longer than that.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1801_09263_gb300", "csrc")


def test_group_is_announced_first(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    exe = tmp_path / "serve_announce_check"
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC,
                        os.path.join(ROOT, "tests", "serve_announce_check.cpp"), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0, out.stdout
