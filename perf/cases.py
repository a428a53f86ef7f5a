"""What a program that uses this framework has it do, as cases that can be timed.

A case is one call (or the few calls a program makes together) at one size:

* ``phi``, ``adj``, ``grad``: the measurement operator on device tensors, its
  adjoint, and both (the data term's residual and gradient through autograd);
* ``psi``: the SARA analysis and synthesis on device tensors;
* ``iter``: iterations of the solver with the image and the blocks' residuals
  read at the end, as an imaging program does between two looks at the image;
* ``group``: the same for several independent problems advanced together.

``listed`` names the sizes, ``draw`` gives others of the same ranges.  Image
sides are those the solver takes (multiples of 16 with 5-smooth grids), the
coverages Gaussian (strongly non-uniform at 0.1 pi, broad at 0.25 pi), the
data blocks radial bands, the data a synthetic sky at 30 dB.

``exact`` computes the same in 64-bit torch from the formulas: Phi = Theta G F
Z with an 8 x 8 Kaiser-Bessel kernel on a 2x grid, Psi = Dirac + db1..db8 with
4 periodic levels over 3, Algorithm 3 with the preconditioned Algorithm 2.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1701_01748_gb300 import ppd, torch_ops

KAPPA, TAU = 1e-4, 0.49
SIDES = sorted(16 * 2 ** a * 3 ** b * 5 ** c for a in range(8) for b in range(5) for c in range(4)
               if 64 <= 16 * 2 ** a * 3 ** b * 5 ** c <= 2048)


def _case(name, kind, L0, L1, M=0, blocks=1, spread=0.1, theta="uniform", iters=0, n_itr=1, fp64=False, problems=1):
    return dict(name=name, kind=kind, L0=L0, L1=L1, M=M, blocks=blocks, spread=spread, theta=theta, iters=iters,
                n_itr=n_itr, fp64=fp64, problems=problems)


def listed():
    return [
        # the smallest call: one prediction of a small field's visibilities, where latency and launches count
        _case("phi_128", "phi", 128, 128, 8192, 1, 0.25),
        # residual and gradient of a data term (a learned or custom solver around the operators), the flagship size
        _case("grad_512", "grad", 512, 512, 524288, 16),
        # a dirty image of a ragged mosaic: rectangular, mixed-radix sides, odd count, per-visibility weights
        _case("adj_960x400", "adj", 960, 400, 1000003, 7, 0.25, "varying"),
        # the residual and gradient of the widest field with 8M visibilities
        _case("grad_4096", "grad", 4096, 4096, 8388608, 256),
        # the prior alone (sparsity of an image, image of a coefficient set): small and large images
        _case("psi_256", "psi", 256, 256),
        _case("psi_2048", "psi", 2048, 2048),
        # imaging: iterations of the solver between two looks at the image, small to large
        _case("iter_128", "iter", 128, 128, 8192, 1, 0.25, iters=50),
        _case("iter_512", "iter", 512, 512, 524288, 16, iters=50),
        _case("iter_1024", "iter", 1024, 1024, 4194304, 64, iters=25),
        # imaging with three inner steps of the ellipsoid projection, rectangular mixed-radix field, per-visibility weights
        _case("iter_640x480_inner3", "iter", 640, 480, 700001, 12, 0.15, "varying", iters=25, n_itr=3),
        # the double-precision solver, which a program uses to check a result
        _case("iter_256_fp64", "iter", 256, 256, 131072, 8, iters=10, fp64=True),
        # a batch of small independent problems (facets, channels) advanced together
        _case("group_8", "group", 128, 256, 0, 4, iters=50, problems=8),
    ]


def draw(rng):
    def logu(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    def side(lo, hi):
        t = logu(lo, hi)
        return min((s for s in SIDES if lo <= s <= hi), key=lambda s: abs(s - t))

    kind = rng.choice(["phi", "adj", "grad", "psi", "iter", "iter", "iter", "group"])
    if kind == "psi":
        return {k: v for k, v in _case("", kind, side(64, 2048), side(64, 2048)).items() if k != "name"}
    if kind == "group":
        lo = side(64, 128)
        c = _case("", kind, lo, side(lo + 16, 320), 0, rng.randint(2, 8), iters=rng.randint(20, 50),
                  problems=rng.randint(3, 8))
        return {k: v for k, v in c.items() if k != "name"}
    fp64 = kind == "iter" and rng.random() < 0.15
    hi = 256 if fp64 else 1024 if kind == "iter" else 2048
    L0 = side(64, hi)
    L1 = L0 if rng.random() < 0.5 else side(64, hi)
    M = int(min(max(500, logu(0.25, 8.0) * L0 * L1), 300000 if fp64 else 4200000)) | 1
    c = _case("", kind, L0, L1, M, rng.randint(1, max(1, min(64, M // 4000))), rng.choice([0.1, 0.15, 0.25]),
              rng.choice(["uniform", "varying"]), iters=(rng.randint(5, 10) if fp64 else rng.randint(10, 40))
              if kind == "iter" else 0, n_itr=rng.choice([1, 1, 3]) if kind == "iter" else 1, fp64=fp64)
    return {k: v for k, v in c.items() if k != "name"}


# ------------------------------------------------------------------ inputs
def _sky(L0, L1, rng):
    """Point sources and Gaussian blobs: (points, blobs) as plain numbers."""
    n = 20
    pts = list(zip(rng.integers(0, L0, n), rng.integers(0, L1, n), 10.0 ** rng.uniform(-3.0, 0.0, n)))
    ls = min(L0, L1)
    blobs = []
    for _ in range(3):
        smaj = rng.uniform(0.03, 0.05) * ls
        blobs.append((rng.uniform(0.3, 0.7) * L0, rng.uniform(0.3, 0.7) * L1, smaj, smaj * rng.uniform(0.3, 1.0),
                      rng.uniform(0.0, math.pi), 10.0 ** rng.uniform(-2.0, -1.0)))
    return pts, blobs


def _image(sky, L0, L1):
    pts, blobs = sky
    r = torch.arange(L0, dtype=torch.float64, device="cuda")[:, None]
    c = torch.arange(L1, dtype=torch.float64, device="cuda")[None, :]
    x = torch.zeros(L0, L1, dtype=torch.float64, device="cuda")
    for c0, c1, sa, sb, t, peak in blobs:
        a = math.cos(t) * (r - c0) + math.sin(t) * (c - c1)
        b = -math.sin(t) * (r - c0) + math.cos(t) * (c - c1)
        x += peak * torch.exp(-0.5 * ((a / sa) ** 2 + (b / sb) ** 2))
    for p0, p1, f in pts:
        x[int(p0), int(p1)] += float(f)
    return x


def _spectrum(sky, om, L0, L1):
    """The sky's visibilities at om (the blobs' analytic spectra; they lie well inside the image)."""
    pts, blobs = sky
    y = torch.zeros(om.shape[0], dtype=torch.complex128, device="cuda")
    w0, w1 = om[:, 0], om[:, 1]
    for p0, p1, f in pts:
        y += torch.polar(torch.full_like(w0, float(f)), -(w0 * (int(p0) - L0 / 2) + w1 * (int(p1) - L1 / 2)))
    for c0, c1, sa, sb, t, peak in blobs:
        q = (sa * (math.cos(t) * w0 + math.sin(t) * w1)) ** 2 + (sb * (-math.sin(t) * w0 + math.cos(t) * w1)) ** 2
        y += torch.polar(peak * 2 * math.pi * sa * sb * torch.exp(-0.5 * q),
                         -(w0 * (c0 - L0 / 2) + w1 * (c1 - L1 / 2)))
    return y


def _problem(L0, L1, M, blocks, spread, theta, seed):
    """One imaging problem's data, on the device."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    sky = _sky(L0, L1, np.random.default_rng(seed))
    om = torch.randn(M, 2, generator=gen, dtype=torch.float64, device="cuda") * (spread * math.pi)
    om = torch.remainder(om + math.pi, 2 * math.pi) - math.pi
    r = om.square().sum(1).sqrt()
    block = torch.clamp((blocks * r / r.max()).floor(), max=blocks - 1).to(torch.int32)
    y = _spectrum(sky, om, L0, L1)
    sigma = float((y.abs().square().mean() * 1e-3).sqrt())
    s = torch.full((M,), sigma, dtype=torch.float64, device="cuda")
    if theta == "varying":
        s = s * torch.exp(0.5 * torch.randn(M, generator=gen, dtype=torch.float64, device="cuda").clamp(-2, 2))
    noise = torch.randn(M, 2, generator=gen, dtype=torch.float64, device="cuda") * (s / math.sqrt(2.0))[:, None]
    return dict(L0=L0, L1=L1, sky=sky, om=om, block=block, y=y + torch.view_as_complex(noise), theta=1.0 / s)


def _eta(p):
    """The data step a program keeps with its coverage: below 1/||U^(1/2) Phi||^2, which is near theta^2 K0 K1."""
    return 1.0 / (1.3 * float(p["theta"].max()) ** 2 * 4 * p["L0"] * p["L1"])


def _solver(p, blocks, n_itr=1, fp64=False):
    s = ppd.Solver(p["L0"], blocks, L1=p["L1"], n_itr=n_itr, eta=_eta(p),
                   precision=ppd.PPD_FP64_PLAIN if fp64 else ppd.PPD_FP32_FP64NORMS)
    return s.set_problem(p["om"].cpu().numpy(), p["y"].cpu().numpy(), p["block"].cpu().numpy(),
                         theta=p["theta"].cpu().numpy())


def _group_sizes(case):
    """(side, visibilities) of the problems of a batch, spread between the case's two sides."""
    k, out = case["problems"], []
    sides = [s for s in SIDES if case["L0"] <= s <= case["L1"]]
    for i in range(k):
        L = sides[i * (len(sides) - 1) // max(1, k - 1)]
        out.append((L, (2 + i % 3) * L * L + 2 * i + 1))
    return out


def _problems(case, seed):
    if case["kind"] == "group":
        return [_problem(L, L, M, case["blocks"], case["spread"], case["theta"], 1000 * seed + i)
                for i, (L, M) in enumerate(_group_sizes(case))]
    return [_problem(case["L0"], case["L1"], case["M"], case["blocks"], case["spread"], case["theta"], 1000 * seed)]


def _psi_inputs(case, seed):
    """An image with some noise, and a set of clipped coefficients as the solver's duals are."""
    L0, L1 = case["L0"], case["L1"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = _image(_sky(L0, L1, np.random.default_rng(seed)), L0, L1)
    x = (x + 1e-3 * torch.randn(L0, L1, generator=gen, dtype=torch.float64, device="cuda")).float()
    c = (2 * KAPPA * torch.randn(9, L0, L1, generator=gen, device="cuda")).clamp(-KAPPA, KAPPA)
    return x, c


def _op_inputs(p):
    """The image whose visibilities are asked for, and whitened visibilities to image."""
    return _image(p["sky"], p["L0"], p["L1"]).float(), (p["theta"] * p["y"]).to(torch.complex64)


class _Group:
    """A batch and its contexts (the group is destroyed before them)."""

    def __init__(self, solvers):
        self.solvers = solvers
        self.handle = ppd.ppd_group_create([s.ctx for s in solvers])

    def __del__(self):
        ppd.ppd_group_destroy(self.handle)
        for s in self.solvers:
            s.close()


def prepare(case, seed):
    kind = case["kind"]
    st = dict(kind=kind, iters=case["iters"])
    if kind == "psi":
        st["x"], st["c"] = _psi_inputs(case, seed)
        st["solver"] = ppd.Solver(case["L0"], 1, L1=case["L1"])
        return st
    ps = _problems(case, seed)
    if kind == "group":
        st["group"] = _Group([_solver(p, case["blocks"]) for p in ps])
        return st
    p = ps[0]
    st["solver"] = _solver(p, case["blocks"], case["n_itr"], case["fp64"])
    if kind != "iter":
        st["x"], st["y"] = _op_inputs(p)
    return st


# ------------------------------------------------------------------ one pass
def _stream():
    return torch.cuda.current_stream().cuda_stream


def _look(s):
    """The image, in the precision the solver holds it."""
    x = s.image()
    return x if s.cfg.precision == ppd.PPD_FP64_PLAIN else x.astype(np.float32)


def run(st):
    kind = st["kind"]
    if kind == "group":
        g = st["group"]
        ppd.ppd_group_iterate(g.handle, st["iters"])
        return [_look(s) for s in g.solvers]
    s = st["solver"]
    if kind == "iter":
        stats = s.iterate(st["iters"])
        res = stats["block_residual"]
        # sums over the solver's arrays, in the precision of those arrays
        return dict(image=_look(s), residual=res if s.cfg.precision == ppd.PPD_FP64_PLAIN else res.astype(np.float32))
    if kind == "psi":
        x, c = st["x"], st["c"]
        coef, img = torch.empty_like(c), torch.empty_like(x)
        ppd.ppd_psi_analysis(s.ctx, x.data_ptr(), coef.data_ptr(), _stream())
        ppd.ppd_psi_synthesis(s.ctx, c.data_ptr(), img.data_ptr(), _stream())
        return dict(coef=coef, image=img)
    if kind == "phi":
        return torch_ops.phi(st["x"], s)
    if kind == "adj":
        y = st["y"]
        img = torch.empty(s.L, s.L1, device="cuda")
        ppd.ppd_op_adjoint(s.ctx, y.data_ptr(), img.data_ptr(), _stream())
        return img
    x = st["x"].detach().requires_grad_()
    r = torch_ops.phi(x, s) - 0.5 * st["y"]
    r.backward(r.detach())
    return dict(residual=r.detach(), grad=x.grad)


# ------------------------------------------------------------------ what a pass cannot do without
def _fft_flops(L0, L1):
    """The 2x padded transform with half of its rows and columns empty."""
    K0, K1 = 2 * L0, 2 * L1
    return 2.5 * L0 * K1 * math.log2(K1) + 5.0 * K1 * K0 * math.log2(K0)


def _psi_flops(N):
    """Both halves of both axes, 8 filters of 2 .. 16 taps, 4 levels (sum of 1/4^l)."""
    return 2 * 2 * 72 * N * 85.0 / 64.0


def work(case):
    kind = case["kind"]
    r = 8 if case["fp64"] else 4
    if kind == "group":
        sizes = [(L, L, M) for L, M in _group_sizes(case)]
    else:
        sizes = [(case["L0"], case["L1"], case["M"])]
    byts = flops = 0.0
    for L0, L1, M in sizes:
        N = L0 * L1
        vis = M * (2 * 8 * 14 + 2 * 2 * 72)   # 16 weights by a degree-7 polynomial, 8 x 8 complex taps row by row
        if kind == "psi":
            byts += 2 * 10 * N * r            # image and 9 coefficient images, each way
            flops += 2 * _psi_flops(N)
        elif kind in ("phi", "adj"):
            byts += M * (3 * r + 2 * r) + N * r   # cell and fractions, the visibility, the image
            flops += vis + _fft_flops(L0, L1)
        elif kind == "grad":
            byts += M * (3 * r + 3 * 2 * r) + 2 * N * r   # as above, the data read and the residual written
            flops += 2 * (vis + _fft_flops(L0, L1))
        else:
            it = case["iters"]
            # record, data, v and p each way; the 9 duals each way, x and xt each way
            byts += it * (M * (4 * r + 2 * r * 5) + N * r * (18 + 4)) + N * r
            flops += it * (2 * (vis + _fft_flops(L0, L1)) + 2 * _psi_flops(N) + case["n_itr"] * 20 * M)
    return {"bytes": byts, "flops": flops}


# ------------------------------------------------------------------ the same in 64 bits
class _Phi:
    """Phi = Theta G F Z and its adjoint in complex128, tap by tap."""

    J, BETA = 8, 2.34 * 8

    def __init__(self, p):
        self.L, self.K = (p["L0"], p["L1"]), (2 * p["L0"], 2 * p["L1"])
        self.theta = p["theta"]
        b = torch.tensor(self.BETA, dtype=torch.float64, device="cuda")
        i0b = torch.special.i0(b)
        self.base, self.frac, self.s, self.at = [], [], [], []
        self.cell = 0
        for ax in (0, 1):
            L, K = self.L[ax], self.K[ax]
            kap = (p["om"][:, ax] * float(K)) * 0.15915494309189535
            f = torch.floor(kap)
            self.base.append(f.long() - 3)
            self.frac.append(kap - f)
            self.cell = self.cell * K + torch.remainder(torch.floor(kap + 0.5).long(), K)
            n = torch.arange(L, dtype=torch.float64, device="cuda") - L // 2
            q = torch.sqrt(b * b - (math.pi * self.J * n / K) ** 2)
            self.s.append(1.0 / (self.J / i0b * torch.sinh(q) / q))
            self.at.append(torch.remainder(torch.arange(L, device="cuda") - L // 2, K))
        self.i0b = i0b

    def _taps(self, lo, hi):
        for a in range(self.J):
            for ax in (0, 1):
                d = (self.frac[ax][lo:hi] + (3 - a)) * 0.25
                t = 1.0 - d * d
                w = torch.where(t >= 0, torch.special.i0(self.BETA * torch.sqrt(t.clamp(min=0))) / self.i0b, 0.0)
                yield ax, a, torch.remainder(self.base[ax][lo:hi] + a, self.K[ax]), w

    def _chunks(self):
        M = self.theta.shape[0]
        for lo in range(0, M, 1 << 20):
            hi = min(M, lo + (1 << 20))
            t = {(ax, a): (i, w) for ax, a, i, w in self._taps(lo, hi)}
            yield lo, hi, [t[0, a] for a in range(self.J)], [t[1, a] for a in range(self.J)]

    def forward(self, x):
        z = torch.zeros(self.K, dtype=torch.complex128, device="cuda")
        z[self.at[0][:, None], self.at[1][None, :]] = (self.s[0][:, None] * self.s[1][None, :] * x).to(z.dtype)
        grid = torch.fft.fft2(z).reshape(-1)
        y = torch.empty(self.theta.shape[0], dtype=torch.complex128, device="cuda")
        for lo, hi, t0, t1 in self._chunks():
            acc = torch.zeros(hi - lo, dtype=torch.complex128, device="cuda")
            for i0, w0 in t0:
                for i1, w1 in t1:
                    acc += (w0 * w1) * grid[i0 * self.K[1] + i1]
            y[lo:hi] = acc
        return self.theta * y

    def adjoint(self, y):
        grid = torch.zeros(self.K[0] * self.K[1], dtype=torch.complex128, device="cuda")
        for lo, hi, t0, t1 in self._chunks():
            v = (self.theta[lo:hi] * y[lo:hi])
            for i0, w0 in t0:
                for i1, w1 in t1:
                    grid.index_add_(0, i0 * self.K[1] + i1, (w0 * w1) * v)
        img = torch.fft.ifft2(grid.reshape(self.K)) * float(self.K[0] * self.K[1])
        return (self.s[0][:, None] * self.s[1][None, :] * img[self.at[0][:, None], self.at[1][None, :]]).real


def _filters():
    """db1 .. db8 by the minimum-phase spectral factorisation (Daubechies 1988), larger end first."""
    out = []
    for p in range(1, 9):
        poly = np.array([1.0 + 0j])
        for _ in range(p):
            poly = np.convolve(poly, [1.0, 1.0])
        for yr in np.roots([math.comb(p - 1 + k, k) for k in range(p)][::-1]):
            a = 1.0 - 2.0 * yr
            s = np.sqrt(a * a - 1.0 + 0j)
            poly = np.convolve(poly, [1.0, -(a + s if abs(a + s) < abs(a - s) else a - s)])
        h = np.real(poly) * (math.sqrt(2.0) / np.real(poly).sum())
        out.append([float(v) for v in (h if abs(h[0]) >= abs(h[-1]) else h[::-1])])
    return out


def _pair(h):
    return h, [(-1.0) ** k * h[len(h) - 1 - k] for k in range(len(h))]


def _ana1(x, h, ax):
    halves = []
    for f in _pair(h):
        acc = 0
        for k, c in enumerate(f):
            r = torch.roll(x, -k, ax)
            acc = acc + c * (r[::2] if ax == 0 else r[:, ::2])
        halves.append(acc)
    return torch.cat(halves, ax)


def _syn1(c, h, ax):
    out = torch.zeros_like(c)
    for part, f in zip(torch.chunk(c, 2, ax), _pair(h)):
        up = torch.zeros_like(c)
        (up[::2] if ax == 0 else up[:, ::2]).copy_(part)
        for k, v in enumerate(f):
            out += v * torch.roll(up, k, ax)
    return out


def _analysis(x, hs):
    out = torch.empty((9,) + tuple(x.shape), dtype=torch.float64, device="cuda")
    out[0] = x
    for i, h in enumerate(hs):
        c = out[i + 1]
        c.copy_(x)
        for lev in range(4):
            n0, n1 = x.shape[0] >> lev, x.shape[1] >> lev
            c[:n0, :n1] = _ana1(_ana1(c[:n0, :n1], h, 1), h, 0)
    return out / 3.0


def _synthesis(c, hs):
    out = c[0].clone()
    for i, h in enumerate(hs):
        x = c[i + 1].clone()
        for lev in range(3, -1, -1):
            n0, n1 = x.shape[0] >> lev, x.shape[1] >> lev
            x[:n0, :n1] = _syn1(_syn1(x[:n0, :n1], h, 0), h, 1)
        out += x
    return out / 3.0


def _solve(p, blocks, iters, n_itr):
    """Algorithm 3 from zero; the image and the residual of the last data step."""
    P, hs, eta = _Phi(p), _filters(), _eta(p)
    blk = p["block"].long()
    cnt = torch.bincount(P.cell, minlength=P.K[0] * P.K[1])
    U = 1.0 / cnt[P.cell].double()
    Mj = torch.bincount(blk, minlength=blocks).double()
    eps = torch.sqrt(Mj + 2.0 * torch.sqrt(Mj)).clamp(min=1.0)
    umax = torch.zeros(blocks, dtype=torch.float64, device="cuda").scatter_reduce_(0, blk, U, "amax")
    muU = U / umax.clamp(min=1e-300)[blk].square()
    yw = P.theta * p["y"]

    def norms(d):
        return torch.zeros(blocks, dtype=torch.float64, device="cuda").index_add_(0, blk, d.abs().square()).sqrt()

    def ball(w):
        n = norms(w - yw)
        c = torch.where(n > eps, eps / n.clamp(min=1e-300), torch.ones_like(n))
        return yw + c[blk] * (w - yw)

    x = torch.zeros(p["L0"], p["L1"], dtype=torch.float64, device="cuda")
    xt, u = x.clone(), torch.zeros(9, p["L0"], p["L1"], dtype=torch.float64, device="cuda")
    v = torch.zeros_like(yw)
    q = res = None
    for _ in range(iters):
        phix = P.forward(xt)
        res = norms(phix - yw)
        z = v / U + phix
        q = ball(z) if q is None else q
        for _ in range(n_itr):
            q = ball(q - muU * (q - z))
        v = U * (z - q)
        u = (u + _analysis(xt, hs)).clamp(-KAPPA, KAPPA)
        xb = (x - TAU * (eta * P.adjoint(v) + _synthesis(u, hs))).clamp(min=0.0)
        x, xt = xb, 2.0 * xb - x
    return x, res


def exact(case, seed):
    kind = case["kind"]
    if kind == "psi":
        x, c = _psi_inputs(case, seed)
        hs = _filters()
        return dict(coef=_analysis(x.double(), hs), image=_synthesis(c.double(), hs))
    if kind in ("iter", "group"):
        if case["iters"] * (case["M"] + 0.5 * case["L0"] * case["L1"]) > 1.5e8:
            return None
        out = [_solve(p, case["blocks"], case["iters"], case["n_itr"]) for p in _problems(case, seed)]
        return [x for x, _ in out] if kind == "group" else dict(image=out[0][0], residual=out[0][1])
    p = _problems(case, seed)[0]
    x, y = _op_inputs(p)
    P = _Phi(p)
    if kind == "phi":
        return P.forward(x.double())
    if kind == "adj":
        return P.adjoint(y.to(torch.complex128))
    r = P.forward(x.double()) - 0.5 * y.to(torch.complex128)
    return dict(residual=r, grad=P.adjoint(r))
