"""The kernels that a plan runs as it is created, at the calls that reach them: whole
groups of every size and pairs left over beside them, angles that do not start at
zero (the bracket below the first angle), prepared rays, every shape of the slant
stack, and calls captured into a CUDA graph."""
import numpy as np
import pytest

import synth
from oracle import bst as ob
from oracle import brute
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


def _uneven(V, rng):
    """Angles that start above zero and end below pi."""
    return np.sort(rng.uniform(0.05, 3.05, V)).astype(np.float32)


def _group(M):
    """Slice pairs of a group: 8 up to M = 512, 4 up to 1024, 2 above."""
    return 8 if M <= 512 else 4 if M <= 1024 else 2


def _grouped(M, N, V, S):
    """Whether a call of S slices runs its whole groups interleaved."""
    pairs = (S + 1) // 2
    return pairs >= _group(M) and (pairs % _group(M) == 0 or pairs * M * (V + N) >= 1 << 23)


# (rays, angles, pad, slices): M = 32, 48, 64, 96, 128, 256, 384, 512 (groups of 8), 768, 1024 (of 4),
# 1536, 2048, 2048, 3072, 4096 (of 2); whole groups, an odd slice count among them
@pytest.mark.parametrize("N,V,alpha,S", [(16, 13, 2, 16), (24, 20, 2, 15), (64, 31, 1, 16), (48, 23, 2, 32),
                                         (64, 33, 2, 15), (128, 40, 2, 16), (192, 64, 2, 16), (256, 75, 2, 31),
                                         (384, 50, 2, 8), (512, 61, 2, 7), (768, 40, 2, 4), (1024, 35, 2, 3),
                                         (2048, 24, 1, 4), (1536, 16, 2, 4), (2048, 21, 2, 3)])
@pytest.mark.parametrize("even", [False, True])
def test_whole_groups(bst, N, V, alpha, S, even):
    assert _grouped(alpha * N, N, V, S) and ((S + 1) // 2) % _group(alpha * N) == 0
    rng = np.random.default_rng(N + V + S)
    theta = synth.uniform_angles(V) if even else _uneven(V, rng)
    assert even or theta[0] > 0.0
    sino = rng.standard_normal((S, V, N)).astype(np.float32)
    g = rng.uniform(0.3, 1.4, alpha * N // 2).astype(np.float32)
    ref = np.stack([ob.fbp(s.astype(np.float64), theta, alpha, g.astype(np.float64)) for s in sino])
    plan = bst.Plan(N, theta, alpha)
    assert plan.forward_config["layout"] == "interleaved"
    for shape in (dict(), dict(max_radix=8, chunk_pairs=_group(alpha * N), pair_fast=0, max_lanes=1)):
        plan.set_forward_config(**shape)
        out = torch.full((S, N, N), float("nan"), device="cuda")
        got = plan.fbp(_cuda(sino), g=_cuda(g), out=out).cpu().numpy()
        assert_parity(got, ref, what=f"N={N} V={V} a={alpha} S={S} even={even} {shape}")


# groups of 8, 4 and 2 with pairs left over, calls just above the line between the two ways
@pytest.mark.parametrize("N,V,alpha,S", [(192, 64, 2, 171), (384, 40, 2, 53), (768, 24, 2, 13)])
def test_pairs_left_over_with_uneven_angles(bst, N, V, alpha, S):
    assert _grouped(alpha * N, N, V, S) and ((S + 1) // 2) % _group(alpha * N)
    rng = np.random.default_rng(N + S)
    theta = _uneven(V, rng)
    sino = rng.standard_normal((S, V, N)).astype(np.float32)
    got = bst.Plan(N, theta, alpha).fbp(_cuda(sino)).cpu().numpy()
    for s in (0, S // 2, S - 12, S - 3, S - 1):
        assert_parity(got[s], ob.fbp(sino[s].astype(np.float64), theta, alpha), what=f"N={N} slice {s} of {S}")


# groups of 8, 4 and 2; the last slice alone in its pair
@pytest.mark.parametrize("N,V,S", [(128, 90, 16), (128, 90, 15), (384, 70, 8), (512, 60, 7), (768, 40, 3), (1024, 50, 4)])
@pytest.mark.parametrize("stages", ["all", "shift", "counts"])
def test_prepared_rays_of_whole_groups(bst, N, V, S, stages):
    assert _grouped(2 * N, N, V, S) and ((S + 1) // 2) % _group(2 * N) == 0
    rng = np.random.default_rng(N + S)
    theta = _uneven(V, rng)
    y = np.stack([synth.ellipse_sinogram(synth.random_ellipses(rng, fov_safe=True), theta, N) for _ in range(S)])
    flat, dark = rng.uniform(9000, 11000, (S, N)), rng.uniform(0, 50, (S, N))
    counts = flat[:, None, :] * np.exp(-y) + dark[:, None, :]
    f32 = lambda a: np.asarray(a, dtype=np.float32).astype(np.float64)  # noqa: E731
    plan = bst.Plan(N, theta, 2)
    kw = dict(shift=-2.3 if stages != "counts" else 0.0)
    if stages == "all":
        kw.update(kb_beta=3.0, kb_halfwidth=0.95)
    rays = y if stages == "shift" else counts
    rows = {} if stages == "shift" else dict(flat=_cuda(flat + dark), dark=_cuda(dark))
    out = torch.full((S, N, N), float("nan"), device="cuda")
    got = plan.fbp_prep(_cuda(rays), out=out, **rows, **kw).cpu().numpy()
    for s in range(S):
        ref = prep.prepared_fbp(f32(rays[s]), theta, flat=f32(flat[s] + dark[s]) if rows else None,
                                dark=f32(dark[s]) if rows else None, shift=kw["shift"], kb_beta=kw.get("kb_beta", 0.0),
                                kb_half=kw.get("kb_halfwidth", 1.0))
        assert_parity(got[s], ref, what=f"N={N} {stages} slice {s} of {S}")


def _slant_shape(N, S, sms):
    """(slices / 4, pixels) a thread of the slant stack, as the launch rule has it."""
    blocks = lambda h, r: -(-N // 32) * -(-N // (4 * r)) * -(-S // (4 * h))  # noqa: E731
    b4 = blocks(1, 4)
    c4, c8 = -(-b4 // sms), -(-blocks(2, 4) // sms)
    if c8 >= 3 and 7 * c8 < 4 * c4:
        return 2, 4
    if 5 * b4 > 12 * sms:
        return 1, 4
    return 1, 2 if blocks(1, 1) > sms else 1


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


# (rays, slices, shape): partial tiles and partial groups of slices, angles that end within a staged batch
@pytest.mark.parametrize("N,V,S,shape", [(96, 13, 7, (1, 1)), (192, 25, 5, (1, 2)), (256, 11, 3, (1, 2)),
                                         (384, 14, 6, (1, 4)), (384, 14, 13, (2, 4)), (512, 13, 15, (2, 4))])
def test_slant_stack_shapes(bst, N, V, S, shape):
    if _slant_shape(N, S, _sms()) != shape:
        pytest.skip("another shape on this number of SMs")
    rng = np.random.default_rng(N + S)
    theta = _uneven(V, rng)
    sino = rng.standard_normal((S, V, N)).astype(np.float32)
    got = bst.Plan(N, theta, 1).brute_backproject(_cuda(sino)).cpu().numpy()
    ref = np.stack([brute.backproject(s.astype(np.float64), theta) for s in sino])
    assert_parity(got, ref, what=f"slant N={N} S={S}")


@pytest.mark.parametrize("N,S,shape", [(64, 1, (1, 1)), (256, 4, (1, 2)), (512, 8, (1, 4)), (512, 16, (2, 4))])
@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_slant_stack_value_that_is_not_finite(bst, N, S, shape, value):
    """It reaches the pixels whose interpolation reads it, in its own slice, and no other."""
    if _slant_shape(N, S, _sms()) != shape:
        pytest.skip("another shape on this number of SMs")
    V, j, i, s = 26, 9, N // 2 + 5, S - 1
    rng = np.random.default_rng(N + S)
    theta = synth.uniform_angles(V)
    sino = rng.standard_normal((S, V, N)).astype(np.float32)
    sino[s, j, i] = value
    got = bst.Plan(N, theta, 1).brute_backproject(_cuda(sino)).cpu().numpy()
    c = np.arange(N) - N // 2
    v = c[None, :] * np.cos(np.float64(theta[j])) + c[:, None] * np.sin(np.float64(theta[j])) + N // 2
    away = np.abs(v - i) > 1.0 + 1e-3
    assert np.isfinite(got[s][away]).all() and not np.isfinite(got[s][np.abs(v - i) < 0.9]).any()
    clean = sino.astype(np.float64)
    clean[s, j, i] = 0.0
    assert_parity(got[s][away], brute.backproject(clean[s], theta)[away], what="pixels away from the sample")
    for o in range(s):
        assert_parity(got[o], brute.backproject(clean[o], theta), what=f"slice {o}")


# one chunk of chained kernels, paired and interleaved; one chunk split over the two lanes; several
# chunks; from M = 2048 on no chaining; `warm`: the plan has been called before the capture
@pytest.mark.parametrize("N,V,S,chunk", [(64, 60, 1, 256), (256, 100, 16, 256), (512, 200, 16, 256),
                                         (512, 200, 37, 4), (1024, 300, 4, 256), (768, 200, 8, 256)])
@pytest.mark.parametrize("warm", [True, False])
@pytest.mark.parametrize("call", ["fbp", "prep"])
def test_captured_call(bst, N, V, S, chunk, warm, call):
    """A call captured into a CUDA graph gives what the call itself gives, on the inputs of each replay."""
    gen = torch.Generator(device="cuda").manual_seed(N + S)
    theta = synth.uniform_angles(V)
    plan = bst.Plan(N, theta, 2).set_forward_config(chunk_pairs=chunk)
    same = bst.Plan(N, theta, 2).set_forward_config(chunk_pairs=chunk)
    pairs = (S + 1) // 2
    if (N, S) in ((512, 16), (1024, 4), (768, 8)):   # one chunk, split
        assert chunk >= pairs and pairs * (2 * N) ** 2 >= 1 << 23
    fresh = lambda: torch.rand((S, V, N), device="cuda", generator=gen) + 0.5  # noqa: E731
    sino, out = fresh(), torch.empty((S, N, N), device="cuda")
    flat = torch.full((S, N), 2.0, device="cuda")

    def run(p, x, y):
        if call == "fbp":
            return p.fbp(x, out=y)
        return p.fbp_prep(x, flat=flat, shift=1.25, kb_beta=2.0, out=y)

    plan.workspace("fwd", plan.workspace_bytes(S), sino.device)
    if warm:
        run(plan, sino, out)
    else:
        run(same, sino, out)   # the kernels are loaded, this plan has made no streams yet
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run(plan, sino, out)
    for _ in range(3):
        sino.copy_(fresh())
        out.fill_(float("nan"))
        graph.replay()
        assert torch.equal(out, run(same, sino, torch.empty_like(out)))
    # the plan's streams serve calls outside the graph as before
    assert torch.equal(out, run(plan, sino, torch.empty_like(out)))


# M = 32, 64, 128 (a column pair of less than a warp), 256 to 512 (groups of 8), 768, 1024 (of 4), 1536, 4096 (of 2)
@pytest.mark.parametrize("N,V", [(16, 13), (32, 70), (64, 45), (48, 100), (128, 333), (192, 64), (256, 300), (384, 90),
                                 (512, 100), (768, 75), (2048, 40)])
def test_a_slice_does_not_depend_on_the_slices_beside_it(bst, N, V):
    """Pairs of slices alone (paired kernels) and in whole groups (interleaved): the same volumes, bit for bit."""
    gen = torch.Generator(device="cuda").manual_seed(N + V)
    theta = synth.uniform_angles(V)
    S = 4 * _group(2 * N)   # two groups
    assert _grouped(2 * N, N, V, S) and not _grouped(2 * N, N, V, 2)
    sino = torch.rand((S, V, N), device="cuda", generator=gen) + 0.5
    flat = torch.full((S, N), 2.0, device="cuda")
    plan = bst.Plan(N, theta, 2)
    calls = (lambda s: plan.fbp(sino[s:s + 2]) if s is not None else plan.fbp(sino),
             lambda s: plan.backproject(sino[s:s + 2]) if s is not None else plan.backproject(sino),
             lambda s: plan.fbp_prep(sino[s:s + 2], flat=flat[s:s + 2], shift=1.5) if s is not None
             else plan.fbp_prep(sino, flat=flat, shift=1.5))
    for call in calls:
        whole = call(None)
        for s in range(0, S, 2):
            assert torch.equal(call(s), whole[s:s + 2]), f"slices {s}, {s + 1}"
