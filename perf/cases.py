"""The work that users of this framework have it do, as measurable cases.

A case is a reconstruction, its transpose, a gradient step, a ragged batch or
the slant-stack comparator at one geometry, through the public entry points of
paper_1704_08364_gb300.  Inputs are made on the GPU from the seed alone:
sinograms of random ellipse phantoms in closed form with measurement noise.
A plan belongs to the state, as a program that reconstructs many volumes of
one geometry keeps it; long volume runs tune it first (Plan.autotune), the
others take the plan as it is created.

The host-resident form (fbp_host) is left out: it is the device-resident path
plus copies over a host link that other jobs share.

exact() restates every operation in 64 bits with plain torch.
"""
import math

import numpy as np
import torch

import paper_1704_08364_gb300 as bst

PHOTONS = 1e4


def listed():
    return [
        # one slice while the user waits, the smallest call (workload single-256)
        dict(name="single-256", kind="fbp", rays=256, angles=256, slices=1, pad=2, even=True, taps=False, tuned=False),
        # a few slices of a small detector, unevenly spaced angles, learned taps, length 3 * 2^a
        dict(name="batch-384", kind="fbp", rays=384, angles=300, slices=8, pad=2, even=False, taps=True, tuned=False),
        # an ordinary volume (workload volume-512)
        dict(name="volume-512", kind="fbp", rays=512, angles=512, slices=512, pad=2, even=True, taps=False, tuned=True),
        # the headline geometry (workload volume-2048), a block of its slices
        dict(name="volume-2048", kind="fbp", rays=2048, angles=2048, slices=64, pad=2, even=True, taps=False,
             tuned=True),
        # plain backprojection, odd angle and slice counts, length 3 * 2^a
        dict(name="backproject-1536", kind="backproject", rays=1536, angles=1201, slices=15, pad=2, even=True,
             taps=False, tuned=False),
        # the volume without padding, for quick looks
        dict(name="volume-2048-pad1", kind="fbp", rays=2048, angles=2048, slices=64, pad=1, even=True, taps=False,
             tuned=True),
        # from photon counts at the paper's beamline geometry: normalization, centering, window
        dict(name="beamline-2048", kind="prep", rays=2048, angles=2000, slices=16, pad=2, even=True, taps=False,
             tuned=False, shift=3.25, window=4.0),
        # the accurate interpolation (Kaiser-Bessel gridding)
        dict(name="kaiser-1024", kind="kaiser", rays=1024, angles=1024, slices=16, pad=2, even=True, taps=False,
             tuned=False, width=6),
        # a training step with learnable taps (workload autograd-1024)
        dict(name="autograd-1024", kind="autograd", rays=1024, angles=1024, slices=16, pad=2, even=True, taps=True,
             tuned=False),
        # the transpose alone, as in an iterative reconstruction
        dict(name="adjoint-512", kind="adjoint", rays=512, angles=400, slices=33, pad=2, even=True, taps=False,
             tuned=False),
        # sinograms of mixed sizes in one launch (workload ragged-64)
        dict(name="ragged-64", kind="ragged", sizes="256,512,768,1024,1536,2048", items=64, pick=3),
        # the slant-stack comparator, filtered
        dict(name="slant-512", kind="slant", rays=512, angles=512, slices=16, pad=2, even=True, taps=True, tuned=False),
    ]


#: rays that a plan of pad factor 2 takes, from small detectors to the largest
RAYS = (64, 96, 128, 192, 256, 384, 512, 768, 1024, 1536, 2048)
#: slices * angles * rays of the largest listed case of each kind
MOST = dict(fbp=64 * 2048 * 2048, backproject=64 * 2048 * 2048, prep=16 * 2000 * 2048, kaiser=16 * 1024 * 1024,
            autograd=16 * 1024 * 1024, adjoint=33 * 1024 * 1024, slant=16 * 512 * 512)


def draw(rng):
    kind = rng.choice(["fbp", "fbp", "fbp", "backproject", "prep", "kaiser", "autograd", "adjoint", "ragged", "slant"])
    if kind == "ragged":
        return dict(kind=kind, sizes=",".join(str(n) for n in sorted(rng.sample((256, 512, 768, 1024, 1536, 2048), 4))),
                    items=rng.randint(8, 64), pick=rng.randint(0, 1 << 20))
    top = dict(kaiser=1024, autograd=1024, adjoint=1024, slant=512).get(kind, 2048)
    rays = rng.choice([n for n in RAYS if n <= top])
    angles = min(2048, max(9, int(rays * math.exp(rng.uniform(math.log(0.4), math.log(1.3))))))
    most = max(1, min(512, MOST[kind] // (rays * max(rays, angles))))
    slices = int(round(math.exp(rng.uniform(0.0, math.log(most)))))
    c = dict(kind=kind, rays=rays, angles=angles, slices=slices, pad=2, even=rng.random() < 0.7,
             taps=rng.random() < 0.4, tuned=False)
    if kind in ("fbp", "backproject"):
        c["pad"] = 1 if rng.random() < 0.25 else 2
        c["tuned"] = slices >= 32 and rng.random() < 0.5
    if kind == "backproject":
        c["taps"] = False
    if kind in ("autograd", "slant"):
        c["taps"] = True
    if kind == "prep":
        c["shift"] = round(rng.uniform(-8.0, 8.0), 3) if rng.random() < 0.8 else 0.0
        c["window"] = round(rng.uniform(2.0, 8.0), 2) if rng.random() < 0.5 else 0.0
    if kind == "kaiser":
        c["width"] = rng.choice([4, 6])
    return c


# ---------------------------------------------------------------------------
# inputs

def _angles(case, seed):
    V = case["angles"]
    if case.get("even", True):
        th = np.arange(V, dtype=np.float64) * (np.pi / V)
    else:  # one angle in each of V equal parts of the half circle
        th = (np.arange(V) + np.random.default_rng(seed).uniform(0.05, 0.95, V)) * (np.pi / V)
    return th.astype(np.float32)


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _phantoms(rng, slices):
    """Random ellipses (cx, cy, a, b, psi, rho) inside the field of view, [K][6][S]: 5 to 20 per slice."""
    K = 20
    a, b = rng.uniform(0.05, 0.4, (2, K, slices))
    r = np.sqrt(rng.uniform(0.0, 1.0, (K, slices))) * (0.95 - np.maximum(a, b))
    phi = rng.uniform(0.0, 2.0 * np.pi, (K, slices))
    rho = rng.uniform(-0.5, 1.0, (K, slices)) * (np.arange(K)[:, None] < rng.integers(5, K + 1, slices)[None, :])
    return np.stack([r * np.cos(phi), r * np.sin(phi), a, b, rng.uniform(0.0, np.pi, (K, slices)), rho], axis=1)


def _projections(ells, theta, N):
    """Closed-form parallel projections [S][V][N] of the ellipses."""
    th = torch.from_numpy(theta).cuda()[None, :, None]
    t = ((torch.arange(N, device="cuda") - N // 2) * (2.0 / N))[None, None, :]
    y = torch.zeros((ells.shape[2], theta.size, N), device="cuda")
    for e in ells:
        cx, cy, a, b, psi, rho = (torch.from_numpy(v.astype(np.float32)).cuda()[:, None, None] for v in e)
        a2 = (a * torch.cos(th - psi)) ** 2 + (b * torch.sin(th - psi)) ** 2
        s = t - (cx * torch.cos(th) + cy * torch.sin(th))
        y.addcmul_(s.square_().neg_().add_(a2).clamp_(min=0.0).sqrt_(), 2.0 * rho * a * b / a2)
    return y


def _images(ells, N):
    """The phantoms themselves [S][N][N]."""
    u = (torch.arange(N, device="cuda") - N // 2) * (2.0 / N)
    img = torch.zeros((ells.shape[2], N, N), device="cuda")
    for e in ells:
        cx, cy, a, b, psi, rho = (torch.from_numpy(v.astype(np.float32)).cuda()[:, None, None] for v in e)
        x, y = u[None, None, :] - cx, u[None, :, None] - cy
        p = (x * torch.cos(psi) + y * torch.sin(psi)) / a
        q = (y * torch.cos(psi) - x * torch.sin(psi)) / b
        img += rho * (p * p + q * q <= 1.0)
    return img


def _sinogram(rng, gen, theta, N, slices, counts=False):
    """Noisy sinograms: of counts (with their flat and dark rows), or additive noise of 1 % of each slice's maximum."""
    y = _projections(_phantoms(rng, slices), theta, N)
    if counts:
        dark = torch.rand((slices, N), device="cuda", generator=gen) * 20.0 + 90.0
        flat = PHOTONS * (0.9 + 0.2 * torch.rand((slices, N), device="cuda", generator=gen)) + dark
        lam = (flat - dark)[:, None, :] * torch.exp(-y)
        return torch.poisson(lam, generator=gen) + dark[:, None, :], flat, dark
    sigma = 0.01 * y.abs().amax(dim=(1, 2), keepdim=True)
    return y.addcmul_(torch.randn(y.shape, device="cuda", generator=gen), sigma)


def _taps(rng, n):
    """Filter taps near a learned apodization: a smooth fall-off with small deviations."""
    g = (0.5 + 0.5 * np.cos(np.pi * np.arange(n) / n)) + 0.05 * rng.standard_normal(n)
    return torch.from_numpy(g.astype(np.float32)).cuda()


def _ragged_sizes(case):
    rng = np.random.default_rng(case["pick"])
    return [int(n) for n in rng.choice([int(v) for v in case["sizes"].split(",")], size=case["items"])]


def _inputs(case, seed):
    rng, gen = np.random.default_rng(seed), _generator(seed)
    kind = case["kind"]
    if kind == "ragged":
        even = lambda V: _angles(dict(angles=V), 0)  # noqa: E731
        return dict(sinos=[_sinogram(rng, gen, even(n), n, 1)[0] for n in _ragged_sizes(case)])
    N, S = case["rays"], case["slices"]
    s = dict(theta=_angles(case, seed))
    if case["taps"]:
        s["g"] = _taps(rng, case["pad"] * N // 2)
    if kind == "adjoint":
        s["vol"] = _images(_phantoms(rng, S), N) + 0.05 * torch.randn((S, N, N), device="cuda", generator=gen)
    elif kind == "prep":
        s["counts"], s["flat"], s["dark"] = _sinogram(rng, gen, s["theta"], N, S, counts=True)
    else:
        if kind == "autograd":
            s["target"] = _images(_phantoms(np.random.default_rng(seed), S), N)
        s["sino"] = _sinogram(rng, gen, s["theta"], N, S)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    if case["kind"] == "ragged":
        sizes = _ragged_sizes(case)
        plans = {n: bst.Plan(n, _angles(dict(angles=n), 0), 2) for n in sorted(set(sizes))}
        s["vols"] = [torch.empty((n, n), device="cuda") for n in sizes]
        s["batch"] = bst.RaggedBatch([plans[n] for n in sizes]).bind(s["sinos"], s["vols"])
        return s
    plan = s["plan"] = bst.Plan(case["rays"], s["theta"], case["pad"])
    if case["kind"] == "kaiser":
        plan.set_gridding("kaiser-bessel", case["width"])
    if case["tuned"]:
        plan.autotune()
    if case["kind"] == "autograd":
        s["sino"].requires_grad_(True)
        s["g"].requires_grad_(True)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "ragged":
        s["batch"].run(use_graph=True)
        return s["vols"]
    plan, g = s["plan"], s.get("g")
    if kind in ("fbp", "kaiser"):
        return plan.fbp(s["sino"], g=g)
    if kind == "backproject":
        return plan.backproject(s["sino"])
    if kind == "prep":
        return plan.fbp_prep(s["counts"], flat=s["flat"], dark=s["dark"], shift=case["shift"],
                             kb_beta=case["window"], kb_halfwidth=1.0, g=g)
    if kind == "adjoint":
        return plan.radon_adjoint(s["vol"], bst.FILTER, g)
    if kind == "slant":
        return plan.brute_backproject(s["sino"], g=g)
    loss = (bst.fbp_autograd(s["sino"], g, plan) - s["target"]).square().sum()
    grad_sino, grad_taps = torch.autograd.grad(loss, (s["sino"], g))
    return dict(loss=loss.detach(), grad_sino=grad_sino, grad_taps=grad_taps)


# ---------------------------------------------------------------------------
# what a pass cannot do without

def _fft(M):
    return 5.0 * M * math.log2(M)


def _fbp_work(N, V, S, M, width=0):
    """Bytes and operations of S slices, two to a complex line: transforms along the rays, the columns and the kept rows,
    and the interpolation (bilinear inside the band, or width x width footprints)."""
    grid = 12.0 * (math.pi / 4) * M * M if not width else 6.0 * width * width * V * (M - 1)
    pair = V * (_fft(M) + 6.0 * M) + M * _fft(M) + grid + N * _fft(M) + 4.0 * N * N
    return 4.0 * S * (V * N + N * N), pair * S / 2


def work(case):
    if case["kind"] == "ragged":
        parts = [_fbp_work(n, n, 1, 2 * n) for n in _ragged_sizes(case)]
        return dict(bytes=sum(p[0] for p in parts), flops=sum(p[1] for p in parts))
    N, V, S, M = case["rays"], case["angles"], case["slices"], case["pad"] * case["rays"]
    if case["kind"] == "slant":
        return dict(bytes=4.0 * S * (V * N + N * N), flops=S * (V * _fft(M) + 4.0 * N * N * V))
    nbytes, flops = _fbp_work(N, V, S, M, case.get("width", 0))
    if case["kind"] == "prep":
        nbytes += 8.0 * S * N
    if case["kind"] == "autograd":  # forward, transpose, the rays' spectrum again, the taps' sums
        nbytes = 4.0 * S * (2 * V * N + N * N)
        flops = 2 * flops + S / 2 * V * (_fft(M) + 4.0 * M)
    return dict(bytes=nbytes, flops=flops)


# ---------------------------------------------------------------------------
# the same operations in 64 bits, plain torch

class _Exact:
    """One geometry: theta (float32, widened), N rays, M = pad N."""

    def __init__(self, theta, N, pad):
        self.th = torch.from_numpy(np.asarray(theta, dtype=np.float64)).cuda()
        self.V, self.N, self.M = self.th.numel(), N, pad * N
        k = torch.arange(self.M, device="cuda")
        self.k = torch.where(k < self.M // 2, k, k - self.M)                   # signed frequency of each index
        self.keep = (torch.arange(N, device="cuda") - N // 2) % self.M         # index of each kept sample
        self._taps = None

    def weight(self, g=None, plain=False):
        """W[|k|] of every index: the taps (ramp: 1), or 1 / sigma_k for plain backprojection; 0 at the Nyquist bin."""
        a = self.k.abs()
        h = self.M // 2
        if plain:
            w = torch.where(a > 0, self.M * (2.0 / self.N) / a.clamp(min=1).double(), 0.0)
        elif g is None:
            w = torch.ones(self.M, dtype=torch.float64, device="cuda")
        else:
            w = g.double()[a.clamp(max=h - 1)]
        return torch.where(a == h, 0.0, w)

    def spectrum(self, y):
        p = torch.zeros((self.V, self.M), dtype=torch.float64, device="cuda")
        p[:, self.keep] = y
        return (2.0 / self.N) * torch.fft.fft(p, dim=-1)

    def taps(self):
        """The four taps (flat index into [V][M], weight) of every Cartesian frequency [M][M], bilinear in (radius, angle)."""
        if self._taps is None:
            V, M, th = self.V, self.M, self.th
            c, r = self.k[None, :].double(), self.k[:, None].double()
            rho = torch.sqrt(c * c + r * r)
            up = (r > 0) | ((r == 0) & (c >= 0))
            ang = torch.atan2(torch.where(up, r, -r), torch.where(up, c, -c))
            kap = torch.where(up, rho, -rho)
            ext = torch.cat([th[-1:] - math.pi, th, th[:1] + math.pi])
            J = torch.searchsorted(th, ang.contiguous(), right=True) - 1
            ft = (ang - ext[J + 1]) / (ext[J + 2] - ext[J + 1])
            K = torch.floor(kap)
            fk = kap - K
            K = K.long()
            self._taps = []
            for dj, dk in ((0, 0), (0, 1), (1, 0), (1, 1)):
                row, b = J + dj, K + dk
                flip = (row < 0) | (row == V)
                row = torch.where(row < 0, V - 1, torch.where(row == V, 0, row))
                b = torch.where(flip, -b, b)
                w = (ft if dj else 1.0 - ft) * (fk if dk else 1.0 - fk)
                w = torch.where((rho < M / 2) & (b.abs() < M // 2), w, 0.0)
                self._taps.append(((row * M + b % M).int(), w))
        return self._taps

    def image(self, X):
        dw = self.N / (2.0 * self.M)
        x = torch.fft.ifft2(X) * (dw * dw * self.M * self.M)
        return x[self.keep][:, self.keep].real

    def from_spectrum(self, Y, w):
        Z = Y * w
        Z[:, 0] = Z[:, 0].mean()
        X = torch.zeros((self.M, self.M), dtype=torch.complex128, device="cuda")
        for idx, wt in self.taps():
            X += wt * Z.reshape(-1)[idx.reshape(-1).long()].reshape(idx.shape)
        return self.image(X)

    def fbp(self, y, w):
        return self.from_spectrum(self.spectrum(y), w)

    def pullback(self, f):
        """Transpose of image(), interpolation and the mean at zero frequency, applied to an image."""
        dw = self.N / (2.0 * self.M)
        x = torch.zeros((self.M, self.M), dtype=torch.float64, device="cuda")
        x[self.keep[:, None], self.keep[None, :]] = f
        X = dw * dw * torch.fft.fft2(x)
        lam = torch.zeros((self.V * self.M, 2), dtype=torch.float64, device="cuda")
        for idx, wt in self.taps():
            lam.index_add_(0, idx.reshape(-1), torch.view_as_real(wt * X).reshape(-1, 2))
        lam = torch.view_as_complex(lam).reshape(self.V, self.M)
        lam[:, 0] = lam[:, 0].mean()
        return lam

    def adjoint(self, lam, w):
        return (2.0 / self.N) * self.M * torch.fft.ifft(lam * w, dim=-1).real[:, self.keep]

    def kaiser(self, ys, w, W):
        """Convolution gridding of the polar samples with a Kaiser-Bessel kernel of width W without its pedestal."""
        M, N, V = self.M, self.N, self.V
        al = M / N
        beta = math.pi * math.sqrt((W / al) ** 2 * (al - 0.5) ** 2 - 0.8)
        i0b = float(np.i0(beta))
        ext = torch.cat([self.th[-1:] - math.pi, self.th, self.th[:1] + math.pi])
        ds = N / (2.0 * M)
        area = ((ext[2:] - ext[:-2]) / 2.0)[:, None] * (ds * ds * self.k.abs().double().clamp(min=0.25))[None, :] * w
        cs, rs = self.k * torch.cos(self.th)[:, None], self.k * torch.sin(self.th)[:, None]

        def axis(x):
            first = torch.floor(x - W / 2.0).long() + 1
            u = [(2.0 * ((first + d) - x) / W) ** 2 for d in range(W)]
            phi = [torch.where(v < 1.0, (torch.special.i0(beta * torch.sqrt((1.0 - v).clamp(min=0.0))) - 1.0) / (i0b - 1.0),
                               0.0) for v in u]
            return [(first + d) % M for d in range(W)], phi

        (ci, cw), (ri, rw) = axis(cs), axis(rs)
        nu = W * math.pi * (torch.arange(N, device="cuda").double() - N // 2) / M
        z2 = beta * beta - nu * nu
        z = torch.sqrt(z2.abs()).clamp(min=1e-9)
        C = W * (torch.where(z2 >= 0, torch.sinh(z), torch.sin(z)) / z - torch.sinc(nu / math.pi)) / (i0b - 1.0)
        out = []
        for y in ys:
            a = self.spectrum(y.double()) * area
            G = torch.zeros((M * M, 2), dtype=torch.float64, device="cuda")
            for dc in range(W):
                for dr in range(W):
                    G.index_add_(0, (ri[dr] * M + ci[dc]).reshape(-1),
                                 torch.view_as_real(a * (cw[dc] * rw[dr])).reshape(-1, 2))
            x = torch.fft.ifft2(torch.view_as_complex(G).reshape(M, M)) * (M * M)
            out.append(x[self.keep][:, self.keep].real / (C[:, None] * C[None, :]))
        return torch.stack(out)

    def slant(self, y, g):
        """Slant-stack backprojection of the rays filtered with |sigma| g."""
        M, N = self.M, self.N
        ds = N / (2.0 * M)
        h = self.weight(g) * ds * self.k.abs().double().clamp(min=0.25)
        p = torch.zeros((y.shape[0], self.V, M), dtype=torch.float64, device="cuda")
        p[..., self.keep] = y.double()
        q = torch.fft.ifft(torch.fft.fft(p) * h).real[..., self.keep]
        q = torch.nn.functional.pad(q, (1, 2))                    # zero outside the detector
        ext = torch.cat([self.th[-1:] - math.pi, self.th, self.th[:1] + math.pi])
        wq = (ext[2:] - ext[:-2]) / 2.0
        i = torch.arange(N, device="cuda").double() - N // 2
        out = torch.zeros((y.shape[0], N, N), dtype=torch.float64, device="cuda")
        for j in range(self.V):
            v = (i[None, :] * torch.cos(self.th[j]) + i[:, None] * torch.sin(self.th[j]) + N // 2).clamp(-1.0, float(N))
            n = torch.floor(v)
            f = v - n
            n = n.long() + 1
            out += wq[j] * (q[:, j, n] * (1.0 - f) + q[:, j, n + 1] * f)
        return out


def exact(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "ragged":
        sizes = _ragged_sizes(case)
        out = [None] * len(sizes)
        for n in sorted(set(sizes)):
            e = _Exact(_angles(dict(angles=n), 0), n, 2)
            for i in (i for i, m in enumerate(sizes) if m == n):
                out[i] = e.fbp(s["sinos"][i].double(), e.weight())
        return out
    e = _Exact(s["theta"], case["rays"], case["pad"])
    g = s.get("g")
    if kind in ("fbp", "backproject"):
        w = e.weight(g, plain=kind == "backproject")
        out = torch.empty((case["slices"], e.N, e.N), dtype=torch.float64, device="cuda")
        for i, y in enumerate(s["sino"]):
            out[i] = e.fbp(y.double(), w)
        return out
    if kind == "prep":
        w, beta, t = e.weight(g), case["window"], (torch.arange(e.N, device="cuda").double() - e.N // 2) * (2.0 / e.N)
        turn = torch.exp(2j * math.pi * case["shift"] / e.M * e.k.double())
        u = t - case["shift"] * (2.0 / e.N)
        win = torch.special.i0(beta * torch.sqrt((1.0 - u * u).clamp(min=0.0))) / float(np.i0(beta)) * (u.abs() <= 1.0)
        out = []
        for y, fl, dk in zip(s["counts"].double(), s["flat"].double(), s["dark"].double()):
            y = -torch.log((y - dk).clamp(min=1e-6) / (fl - dk).clamp(min=1e-6))
            out.append(e.from_spectrum(e.spectrum(y * win if beta > 0.0 else y) * turn, w))
        return torch.stack(out)
    if kind == "kaiser":
        return e.kaiser(s["sino"], e.weight(g), case["width"])
    if kind == "slant":
        return e.slant(s["sino"], g)
    if kind == "adjoint":
        return torch.stack([e.adjoint(e.pullback(f.double()), e.weight(g)) for f in s["vol"]])
    w, loss, grads = e.weight(g), 0.0, []
    gg = torch.zeros(e.M // 2, dtype=torch.float64, device="cuda")
    for y, f in zip(s["sino"].double(), s["target"].double()):
        Y = e.spectrum(y)
        R = e.from_spectrum(Y.clone(), w) - f
        loss = loss + R.square().sum()
        lam = e.pullback(2.0 * R)
        grads.append(e.adjoint(lam, w))
        b = (lam.conj() * Y).real.sum(dim=0)
        a = e.k.abs()
        gg.index_add_(0, a[a < e.M // 2], b[a < e.M // 2])
    return dict(loss=loss, grad_sino=torch.stack(grads), grad_taps=gg)
