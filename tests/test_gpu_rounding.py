"""Rounding of fixed coefficients in the FP32 path.  A coefficient that every
visibility, pixel or iteration shares shifts the whole result when it is
rounded, where the rounding of data averages out; these tests measure the
shift of the amplitude against 64-bit values, or the error it causes."""
from __future__ import annotations

import math

import numpy as np
import pytest
import torch

from oracle import nufft
from paper_1701_01748_gb300 import ppd

pytestmark = pytest.mark.gpu


def operator(om, L0, L1):
    M = om.shape[0]
    return ppd.Solver(L0, 1, L1=L1, eta=1.0).set_problem(om, np.zeros(M, complex), np.zeros(M, np.int32))


def coverage(M, seed, spread=0.25):
    om = np.random.default_rng(seed).normal(0, spread * math.pi, (M, 2))
    return np.remainder(om + math.pi, 2 * math.pi) - math.pi


def stream():
    return torch.cuda.current_stream().cuda_stream


def test_weights_keep_the_amplitude():
    """Of a point at the centre the transform is constant, exactly so in FP32
    (sums with zeros), and a visibility is that constant times the sums of its
    taps' weights.  Rounding of data is within 1e-7 per visibility and averages
    to 1e-9 over 20000; the weights' constant terms rounded to FP32 made it
    4e-8 low."""
    L, M = 64, 20000
    om = coverage(M, 1)
    s = operator(om, L, L)
    x = torch.zeros(L, L, device="cuda")
    x[L // 2, L // 2] = 1.0
    y = torch.empty(M, 2, device="cuda")
    ppd.ppd_op_forward(s.ctx, x.data_ptr(), y.data_ptr(), stream())
    z = np.float32(1.0 / nufft.kb_transform(0.0))
    want = np.full(M, float(z * z))
    for ax in (0, 1):
        kap = om[:, ax] * (2 * L / (2 * math.pi))
        frac = kap - np.floor(kap)
        want *= sum(nufft.kb_kernel(frac + 3 - j) for j in range(8))
    err = y.cpu().double().numpy()[:, 0] / want - 1
    assert abs(err.mean()) <= 1e-8
    s.close()


def test_step_keeps_tau_eta():
    """From x = 0 the first iterate is max(0, -tau eta g).  Two steps 2^-24
    apart (less than FP32 resolves in eta or in tau eta) give images apart by
    that factor on average: a pixel's rounding is within 2^-24, its mean over
    the 2000 positive pixels within 2e-9."""
    L, M = 64, 20000
    om = coverage(M, 2)
    rng = np.random.default_rng(2)
    y = rng.normal(size=M) + 1j * rng.normal(size=M)
    img = []
    for eta in (1e-6, 1e-6 * (1 + 2.0 ** -24)):
        s = ppd.Solver(L, 1, eta=eta).set_problem(om, y, np.zeros(M, np.int32))
        s.iterate(1)
        img.append(s.image())
        s.close()
    on = img[0] > 0
    assert on.sum() > 1000
    assert abs((img[1][on] / img[0][on]).mean() - 1 - 2.0 ** -24) <= 1e-8


def adjoint(L0, L1, M, seed):
    """Phi^dagger of ten points' visibilities, and its 64-bit value."""
    om = coverage(M, seed)
    rng = np.random.default_rng(seed)
    at = np.stack([rng.integers(0, L0, 10) - L0 // 2, rng.integers(0, L1, 10) - L1 // 2])
    y = np.exp(-1j * (om @ at)).sum(1).astype(np.complex64)
    s = operator(om, L0, L1)
    yd = torch.from_numpy(y).cuda()
    out = torch.empty(L0, L1, device="cuda")
    ppd.ppd_op_adjoint(s.ctx, yd.data_ptr(), out.data_ptr(), stream())
    got = out.cpu().double().numpy()
    s.close()
    return got, nufft.phi_adjoint(y.astype(np.complex128), nufft.Plan(om, L0, L1))


def test_mixed_radix_adjoint_inverts_single_rows():
    """Rows of length 1440: inverting two real rows in one complex transform
    has the rounding of a complex transform, where the real part of a single
    row's has half of it.  Of the transforms alone, emulated in FP32 on three
    such problems, that is 1.18e-7 against 0.94e-7; with 5e-8 for the gridding
    1.28e-7 and 1.07e-7: the bound is between them."""
    err = []
    for seed in range(6):
        got, ref = adjoint(32, 720, 60000, seed)
        err.append(np.linalg.norm(got - ref) / np.linalg.norm(ref))
    assert np.mean(err) <= 1.17e-7


def test_radix_constants_keep_the_amplitude():
    """Transforms of length 800 (two radix-10 stages an axis): the rounding of
    sin and cos of 2 pi/5 alone shifted the adjoint's amplitude by 1.9e-8; the
    twiddles and the pixel scalings, which differ along a transform, leave a
    few 1e-9."""
    got, ref = adjoint(400, 400, 100000, 5)
    assert abs((got * ref).sum() / (ref ** 2).sum() - 1) <= 1e-8
