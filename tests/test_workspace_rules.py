"""The sizes of a plan's workspaces: what they may grow to and what they shrink to
where memory is short (host code only, no GPU)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")


def test_workspace_sizes_are_bounded(tmp_path):
    """tests/workspace_check.cu: the chunk that a plan starts with."""
    nvcc = NVCC if os.path.exists(NVCC) else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not available")
    exe = tmp_path / "workspace_check"
    r = subprocess.run([nvcc, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1704_08364_gb300", "csrc"),
                        "-I", os.path.join(ROOT, "include"), "-x", "cu",
                        os.path.join(ROOT, "tests", "workspace_check.cu"), "-o", str(exe)],
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and out.stdout.strip() == "OK", out.stdout + out.stderr
