"""The sizes of a plan's workspaces: what they may grow to and what they shrink to
where memory is short (host code only, no GPU)."""
import ctypes
import gc
import os
import shutil
import subprocess

import pytest

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")


def test_workspace_sizes_are_bounded(tmp_path):
    """tests/workspace_check.cu: the chunk that a plan starts with, what the autotuner
    allocates, and the pairs that the adjoint has in flight."""
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


class FakeLib:
    """The calls of libbst that the forward workspace is sized with: two lanes of
    chunk_pairs pairs, 1000 bytes a pair."""

    def __init__(self):
        self.config = [16, 2, 8, 1, 2, 1]

    def bst_workspace_bytes(self, h, slices):
        return 2000 * min(self.config[2], (slices + 1) // 2)

    def bst_plan_get_forward_config(self, h, ref):
        for (name, _), v in zip(type(ref._obj)._fields_, self.config):
            setattr(ref._obj, name, v)
        return 0

    def bst_plan_set_forward_config(self, h, ref):
        self.config = [getattr(ref._obj, name) for name, _ in type(ref._obj)._fields_]
        return 0


@pytest.mark.parametrize("room,slices,pairs", [(1 << 20, 64, 8), (15999, 64, 4), (7000, 64, 2), (2000, 64, 1),
                                               (5000, 6, 1), (5000, 5, 1), (12000, 12, 8), (11999, 11, 3)])
def test_forward_workspace_gives_way_to_little_memory(monkeypatch, room, slices, pairs):
    """A workspace that cannot be allocated is tried with fewer pairs a chunk."""
    from paper_1704_08364_gb300 import api
    plan = api.Plan.__new__(api.Plan)
    plan._h, plan._lib, plan._ws = ctypes.c_void_p(), FakeLib(), {}

    def empty(n, dtype, device):
        if n > room:
            raise torch.OutOfMemoryError("out of memory")
        return torch.zeros(n, dtype=dtype, device=device)

    monkeypatch.setattr(api.torch, "empty", empty)
    def ask():
        try:
            return plan.workspace("fwd", plan._lib.bst_workspace_bytes(None, slices), "cpu")
        except torch.OutOfMemoryError:
            return plan._smaller_workspace("fwd", plan._lib.bst_workspace_bytes, slices, "cpu")

    ws = ask()
    assert ws.numel() == plan._lib.bst_workspace_bytes(None, slices) <= room
    assert plan.forward_config["chunk_pairs"] == pairs
    room = 1999   # not even one pair a lane
    with pytest.raises(torch.OutOfMemoryError):
        plan._ws.clear()
        ask()


@pytest.mark.gpu
def test_calls_go_on_with_smaller_chunks_where_memory_is_short():
    """The forward calls with room for one pair a lane only, by the caching
    allocator's limit for the process."""
    import numpy as np
    import paper_1704_08364_gb300 as bst
    N, V, S = 1024, 1000, 40
    theta = (np.arange(V) * np.pi / V).astype(np.float32)

    def drop_cached():   # and no tensor in a part of a segment whose rest the allocator could still use
        gc.collect()
        torch.cuda.synchronize()
        torch.cuda.empty_cache()

    drop_cached()
    sino = torch.randn((S, V, N), device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    out, ref = torch.empty((S, N, N), device="cuda"), torch.empty((S, N, N), device="cuda")
    bst.Plan(N, theta, 2).fbp(sino, out=ref)
    plan = bst.Plan(N, theta, 2)
    assert plan.forward_config["chunk_pairs"] > 2 and plan.workspace_bytes(S) > 400 << 20
    drop_cached()
    total = torch.cuda.get_device_properties(0).total_memory
    try:
        torch.cuda.set_per_process_memory_fraction((torch.cuda.memory_reserved() + (100 << 20)) / total)
        plan.fbp(sino, out=out)
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    assert plan.forward_config["chunk_pairs"] == 1
    assert torch.allclose(out, ref, rtol=0, atol=float(ref.abs().max()) * 1e-5)
