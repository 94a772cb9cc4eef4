"""The interleaved layout of the forward path (groups of 2 to 8 slice pairs
point by point) gives the oracle's result: FFT lengths at the ends of every
group size, both pad factors and radix schedules, odd angle counts, slice counts
that fill groups exactly, leave pairs over or leave half a pair, and a workspace
that only the packed layout can read."""
import ctypes

import numpy as np
import pytest

import synth
from oracle import bst as ob
from oracle import prep
from gpu_util import assert_parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bst():
    import paper_1704_08364_gb300 as m
    return m


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


# (rays, angles, pad, slices): M = 16 (no groups), 32 (groups of eight pairs, one
# warp a block), 48, 96, 512, 384, 768, 1024, 1536, 2048, 2048, 3072, 4096
@pytest.mark.parametrize("N,V,alpha,S", [(8, 9, 2, 17), (16, 13, 2, 16), (32, 31, 1, 33), (24, 20, 2, 19), (96, 41, 1, 32),
                                         (256, 75, 2, 17), (192, 64, 2, 35), (384, 50, 2, 8), (512, 61, 2, 11),
                                         (768, 40, 2, 6), (1024, 35, 2, 5), (2048, 24, 1, 9), (1536, 16, 2, 4),
                                         (2048, 21, 2, 5)])
def test_interleaved_matches_the_oracle(bst, N, V, alpha, S):
    rng = np.random.default_rng(N + V + S)
    theta = synth.uniform_angles(V) if N != 192 else np.sort(rng.uniform(0.02, 3.1, V)).astype(np.float32)
    sino = rng.standard_normal((S, V, N)).astype(np.float32)
    g = rng.uniform(0.3, 1.4, alpha * N // 2).astype(np.float32)
    plan = bst.Plan(N, theta, alpha)
    ref = np.stack([ob.fbp(s.astype(np.float64), theta, alpha, g.astype(np.float64)) for s in sino])
    for r in (16, 8):
        for chunk, pf, lanes in ((256, 0, 1), (8, 1, 2), (3, 0, 2)):
            plan.set_forward_config(layout="interleaved", max_radix=r, chunk_pairs=chunk, pair_fast=pf, max_lanes=lanes)
            out = torch.full((S, N, N), float("nan"), device="cuda")
            got = plan.fbp(_cuda(sino), g=_cuda(g), out=out).cpu().numpy()
            assert_parity(got, ref, what=f"N={N} V={V} a={alpha} S={S} r={r} chunk={chunk}")


def test_backprojection_and_prepared_rays(bst):
    """Plain backprojection, and bst_fbp_prep (normalization, centering by a
    fraction of a sample, window) on interleaved groups."""
    N, V, S = 128, 90, 18
    rng = np.random.default_rng(5)
    theta = synth.uniform_angles(V)
    y = np.stack([synth.ellipse_sinogram(synth.random_ellipses(rng, fov_safe=True), theta, N) for _ in range(S)])
    plan = bst.Plan(N, theta, 2)
    assert plan.forward_config["layout"] == "interleaved"
    got = plan.backproject(_cuda(y)).cpu().numpy()
    assert_parity(got, np.stack([ob.backproject(s.astype(np.float32).astype(np.float64), theta) for s in y]), what="bp")
    flat, dark = rng.uniform(9000, 11000, (S, N)), rng.uniform(0, 50, (S, N))
    counts = flat[:, None, :] * np.exp(-y) + dark[:, None, :]
    f32 = lambda a: np.asarray(a, dtype=np.float32).astype(np.float64)  # noqa: E731
    got = plan.fbp_prep(_cuda(counts), flat=_cuda(flat + dark), dark=_cuda(dark), shift=-2.3, kb_beta=3.0,
                        kb_halfwidth=0.95).cpu().numpy()
    for s in range(S):
        ref = prep.prepared_fbp(f32(counts[s]), theta, flat=f32(flat[s] + dark[s]), dark=f32(dark[s]), shift=-2.3,
                                kb_beta=3.0, kb_half=0.95)
        assert_parity(got[s], ref, what=f"prep slice {s}")


@pytest.mark.parametrize("N,S", [(64, 4), (256, 16)])
def test_workspace_aligned_to_eight_bytes(bst, N, S):
    """The C ABI asks no more of the workspace than the packed layout needs."""
    from paper_1704_08364_gb300 import _lib
    rng = np.random.default_rng(N)
    V = N // 2 + 1
    theta = synth.uniform_angles(V)
    sino = rng.standard_normal((S, V, N)).astype(np.float32)
    plan = bst.Plan(N, theta, 2)
    nb = plan.workspace_bytes(S)
    ws = torch.empty(nb + 64, dtype=torch.uint8, device="cuda")
    d, out = _cuda(sino), torch.full((S, N, N), float("nan"), device="cuda")
    p = lambda t, o=0: ctypes.c_void_p(t.data_ptr() + o)  # noqa: E731
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert _lib.load().bst_fbp(plan.handle, p(d), S, None, p(out), p(ws, 8), nb, st) == 0
    assert_parity(out.cpu().numpy(), np.stack([ob.fbp(s.astype(np.float64), theta) for s in sino]), what=f"N={N}")


@pytest.mark.parametrize("N,V,alpha,S", [(128, 60, 2, 349), (64, 50, 2, 1150), (384, 40, 2, 53), (768, 24, 2, 13)])
def test_groups_and_pairs_left_over(bst, N, V, alpha, S):
    """Calls large enough for groups although pairs are left over, and slices of
    every kind of them (first group, last group, left over) against the oracle."""
    M, pairs = alpha * N, (S + 1) // 2
    assert pairs * M * (V + N) >= 1 << 23 and pairs % (8 if M <= 512 else 4 if M <= 1024 else 2)
    rng = np.random.default_rng(N + S)
    theta = synth.uniform_angles(V)
    sino = rng.standard_normal((S, V, N)).astype(np.float32)
    plan = bst.Plan(N, theta, alpha)
    plan.set_forward_config(layout="interleaved", chunk_pairs=256)
    got = plan.fbp(_cuda(sino)).cpu().numpy()
    for s in (0, 7, S // 2, S - 18, S - 3, S - 2, S - 1):
        if s >= 0:
            assert_parity(got[s], ob.fbp(sino[s].astype(np.float64), theta, alpha), what=f"N={N} slice {s} of {S}")
    plan.set_forward_config(layout="paired")
    assert_parity(got, plan.fbp(_cuda(sino)).cpu().numpy(), what=f"N={N} paired")
