"""Launch geometry of the batched Cholesky (no GPU): csrc/chol_window.h, compiled with the host
compiler together with tests/chol_window_check.cpp.  A window of 363 tiles has 65,703 pairs
of block rows below its first column, more than a launch's y dimension."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_cholesky_launch_geometry(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "chol_window_check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-o", exe, os.path.join(ROOT, "tests", "chol_window_check.cpp")],
                   check=True, capture_output=True, text=True)
    p = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert p.returncode == 0 and "ALL OK" in p.stdout, p.stdout + p.stderr
