"""Registers and spills of the kernels that a plan uses as it is created, read from
ptxas at compile time, and the slot map of their spectrum layout; no GPU needed.
Blocks of 512 threads run two an SM and blocks of 1024 alone at 64 registers a
thread; Kaiser-Bessel gridding runs 512 threads an SM at 128."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
CSRC = os.path.join(ROOT, "paper_1704_08364_gb300", "csrc")
FLAGS = ["-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include")]


@pytest.fixture(scope="module")
def nvcc():
    exe = NVCC if os.path.exists(NVCC) else shutil.which("nvcc")
    if not exe:
        pytest.skip("nvcc not available")
    return exe


def _ptxas(nvcc, src, out):
    """(registers, bytes of spill stores) by the mangled name of each kernel of src."""
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", *FLAGS, "-Xptxas", "-v",
                        "-c", src, "-o", str(out)], capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout + r.stderr
    res = {}
    for block in (r.stdout + r.stderr).split("Compiling entry function")[1:]:
        name = re.match(r"\s*'([^']*)'", block).group(1)
        res[name] = (int(re.search(r"Used (\d+) registers", block).group(1)),
                     int(re.search(r"(\d+) bytes spill stores", block).group(1)))
    return res


def test_default_forward_kernels_do_not_spill(nvcc, tmp_path):
    res = _ptxas(nvcc, os.path.join(ROOT, "tests", "kernel_resources_default.cu"), tmp_path / "k.o")
    for kernel, count, most in (("k_ray_inter", 6, 64), ("k_grid_inter", 3, 64), ("k_row_inter", 3, 64),
                                ("kb_unit", 2, 128)):
        found = {n: v for n, v in res.items() if re.search(r"\d" + kernel + "ILi", n)}
        assert len(found) == count, (kernel, sorted(res))
        for n, (regs, spill) in found.items():
            assert regs <= most and spill == 0, f"{n}: {regs} registers, {spill} bytes spilled"


def test_adjoint_kernels_spill_no_more_than_they_do(nvcc, tmp_path):
    """Two blocks of 512 threads (or as many threads in smaller ones) an SM: 64
    registers, which the polar stage of four pairs exceeds by up to 144 bytes; the
    transforms and the filter gradient spill nothing."""
    res = _ptxas(nvcc, os.path.join(CSRC, "adjoint.cu"), tmp_path / "a.o")
    polar = {n: v for n, v in res.items() if "k_adj_polar" in n}
    assert len(polar) >= 40
    for n, (regs, spill) in polar.items():
        pairs = int(re.search(r"k_adj_polarILi\d+ELi\d+ELi\d+ELi(\d)E", n).group(1))
        assert spill <= (144 if pairs == 4 else 8), f"{n}: {regs} registers, {spill} bytes spilled"
    for n, (regs, spill) in res.items():
        if re.search("k_adj_row_fft|k_adj_col_fft|k_fg_ray", n):
            assert spill == 0, f"{n}: {regs} registers, {spill} bytes spilled"


def test_interleaved_layout_slot_map_is_a_bijection(nvcc, tmp_path):
    exe = tmp_path / "inter_layout_check"
    r = subprocess.run([nvcc, *FLAGS, "-O2", "-x", "cu", os.path.join(ROOT, "tests", "inter_layout_check.cu"),
                        "-o", str(exe)], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and out.stdout.strip() == "OK", out.stdout + out.stderr
