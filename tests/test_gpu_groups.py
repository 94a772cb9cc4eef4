"""Kernels that take several slices at once, at the slice counts where groups
begin and end: the adjoint and the filter gradient (up to four pairs, and what
remains of them), Kaiser-Bessel gridding (the same) and the slant stack (four or
eight slices, one or four pixels a thread), against the oracle."""
import numpy as np
import pytest

import synth
from oracle import adjoint as oa
from oracle import bst as ob
from oracle import brute
from oracle import kb
from gpu_util import assert_parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bst():
    import paper_1704_08364_gb300 as m
    return m


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def _angles(V, rng, even):
    return synth.uniform_angles(V) if even else np.sort(rng.uniform(0.02, 3.1, V)).astype(np.float32)


# M = 16, 48, 128, 192 (rows filling a warp), 512, 1536 (128 threads a line), 3072 (groups of two)
@pytest.mark.parametrize("N,V,alpha,even", [(8, 9, 2, True), (24, 10, 2, False), (128, 33, 1, True), (96, 21, 2, False),
                                             (256, 30, 2, True), (768, 11, 2, True), (1536, 5, 2, True)])
@pytest.mark.parametrize("S", [1, 5, 8, 13])
def test_adjoint_and_filter_gradient_groups(bst, N, V, alpha, even, S):
    if S > 5 and N > 700:
        pytest.skip("the smaller lengths cover it")
    rng = np.random.default_rng(N + S)
    theta = _angles(V, rng, even)
    p = rng.standard_normal((S, V, N)).astype(np.float32)
    f = rng.standard_normal((S, N, N)).astype(np.float32)
    g = rng.uniform(0.3, 1.5, alpha * N // 2).astype(np.float32)
    plan = bst.Plan(N, theta, alpha)
    gp, gg = plan.fbp_backward(_cuda(p), _cuda(f), _cuda(g))
    d = lambda a: a.astype(np.float64)  # noqa: E731
    ref = np.stack([oa.bst_adjoint(d(x), theta, alpha, "filter", d(g)) for x in f])
    assert_parity(gp.cpu().numpy(), ref, what=f"grad p N={N} S={S}")
    assert_parity(gg.cpu().numpy(), sum(oa.filter_grad(d(p[s]), d(f[s]), theta, alpha) for s in range(S)),
                  what=f"grad g N={N} S={S}")


# strips wrap at both ends; M = 16 with the widest kernel, M >= 3072 in groups of two
@pytest.mark.parametrize("N,V,alpha,W,even", [(8, 7, 2, 8, True), (24, 16, 2, 2, False), (96, 40, 2, 6, False),
                                               (128, 64, 2, 4, True), (1536, 6, 2, 6, True)])
@pytest.mark.parametrize("S", [2, 4, 6, 14])
def test_kaiser_bessel_groups(bst, N, V, alpha, W, even, S):
    if N > 700 and S > 6:
        pytest.skip("the smaller lengths cover it")
    rng = np.random.default_rng(N + S + W)
    theta = _angles(V, rng, even)
    sino = rng.standard_normal((S, V, N)).astype(np.float32)
    plan = bst.Plan(N, theta, alpha).set_gridding("kaiser-bessel", W)
    got = plan.fbp(_cuda(sino)).cpu().numpy()
    ref = np.stack([kb.kb_fbp(s.astype(np.float64), theta, alpha, width=W) for s in sino])
    assert_parity(got, ref, what=f"KB N={N} W={W} S={S}")


# both sides of the lines between one and four pixels a thread, four and eight
# slices; angle counts around the staged batch
@pytest.mark.parametrize("N,V,S", [(32, 11, 1), (48, 12, 4), (96, 13, 5), (512, 25, 4), (512, 25, 9), (384, 12, 40)])
def test_slant_stack_groups(bst, N, V, S):
    rng = np.random.default_rng(N + S)
    theta = _angles(V, rng, S % 2 == 1)
    sino = rng.standard_normal((S, V, N)).astype(np.float32)
    got = bst.Plan(N, theta, 1).brute_backproject(_cuda(sino)).cpu().numpy()
    ref = np.stack([brute.backproject(s.astype(np.float64), theta) for s in sino])
    assert_parity(got, ref, what=f"slant N={N} S={S}")


@pytest.mark.parametrize("S", [1, 8])
def test_slant_stack_keeps_a_value_that_is_not_finite_to_its_own_pixels(bst, S):
    """An infinite sample reaches the pixels whose interpolation reads it and no other."""
    N, V = 512, 26
    rng = np.random.default_rng(1)
    theta = synth.uniform_angles(V)
    sino = rng.standard_normal((S, V, N)).astype(np.float32)
    j, i = 9, 300
    sino[0, j, i] = np.inf
    got = bst.Plan(N, theta, 1).brute_backproject(_cuda(sino)).cpu().numpy()
    c = np.arange(N) - N // 2
    v = c[None, :] * np.cos(np.float64(theta[j])) + c[:, None] * np.sin(np.float64(theta[j])) + N // 2
    away = np.abs(v - i) > 1.0 + 1e-3
    assert np.isfinite(got[0][away]).all() and not np.isfinite(got[0][np.abs(v - i) < 0.9]).any()
    clean = sino.astype(np.float64)
    clean[0, j, i] = 0.0
    assert_parity(got[0][away], brute.backproject(clean[0], theta)[away], what="pixels away from the sample")


# first passes of radix 3, 6 and 12 (their lines are padded differently), then 16 or
# less: M = 48, 48, 96, 192, 384, 768, 1536, 3072
@pytest.mark.parametrize("N,V,alpha", [(24, 9, 2), (48, 20, 1), (48, 31, 2), (192, 16, 1), (192, 33, 2), (384, 30, 2),
                                        (768, 20, 2), (1536, 9, 2)])
@pytest.mark.parametrize("layout", ["packed", "paired"])
def test_lengths_with_a_factor_of_three(bst, N, V, alpha, layout):
    rng = np.random.default_rng(N + V)
    theta = _angles(V, rng, V % 2 == 0)
    sino = rng.standard_normal((3, V, N)).astype(np.float32)
    ref = np.stack([ob.fbp(s.astype(np.float64), theta, alpha) for s in sino])
    plan = bst.Plan(N, theta, alpha)
    for r in (16, 8):
        for xchg in (0, 1):
            plan.set_forward_config(layout=layout, max_radix=r, chunk_pairs=2, grid_xchg=xchg)
            assert_parity(plan.fbp(_cuda(sino)).cpu().numpy(), ref, what=f"{layout} N={N} a={alpha} r={r}")
