"""The loop over host threads that builds plan tables (no GPU)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_threads_that_cannot_be_started_leave_no_index_out(tmp_path):
    """Every allocation of a starting thread fails once: no abort, no index lost."""
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    exe = tmp_path / "parallel_check"
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I",
                        os.path.join(ROOT, "paper_1704_08364_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "parallel_check.cpp"), "-o", str(exe)],
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and out.stdout.strip() == "OK", out.stdout + out.stderr
