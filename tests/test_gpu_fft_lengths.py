"""Phi and Phi^dagger against the FP64 oracle with every FFT length class on
either axis: each power of two (register core, row and column layouts of both
precisions), and lengths whose plans use each radix of the mixed-radix core.
Tolerances of the operator tests (1e-5 in FP32, 1e-10 in FP64)."""
from __future__ import annotations

import math

import numpy as np
import pytest
import torch

from oracle import nufft
from paper_1701_01748_gb300 import ppd

pytestmark = pytest.mark.gpu

F32, F64 = ppd.PPD_FP32_FP64NORMS, ppd.PPD_FP64_PLAIN


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def op_forward(s, x, dt):
    xd = torch.tensor(x, dtype=dt, device="cuda")
    yd = torch.empty((s.M, 2), dtype=dt, device="cuda")
    ppd.ppd_op_forward(s.ctx, xd.data_ptr(), yd.data_ptr(), torch.cuda.current_stream().cuda_stream)
    return yd.cpu().double().numpy() @ np.array([1.0, 1j])


def op_adjoint(s, y, dt):
    yd = torch.tensor(np.stack([y.real, y.imag], 1), dtype=dt, device="cuda")
    xd = torch.empty((s.L, s.L1), dtype=dt, device="cuda")
    ppd.ppd_op_adjoint(s.ctx, yd.data_ptr(), xd.data_ptr(), torch.cuda.current_stream().cuda_stream)
    return xd.cpu().double().numpy()


SIDES = [16, 32, 48, 64, 80, 96, 128, 144, 160, 240, 256, 400, 432, 512, 640, 960, 1024, 2000, 2048, 3888, 4096]


@pytest.mark.parametrize("prec", [F32, F64])
@pytest.mark.parametrize("n", SIDES)
def test_length_on_either_axis(n, prec):
    if prec == F64 and n == 3888:
        pytest.skip("FP64 mixed-radix lengths end at 4096")
    tol, dt = (1e-5, torch.float32) if prec == F32 else (1e-10, torch.float64)
    rng = np.random.default_rng(n)
    for L0, L1 in ((n, 16), (16, n), (48, n)) if n < 2000 else ((n, 16), (16, n)):
        M = 300
        om = rng.uniform(-math.pi, math.pi, (M, 2))
        s = ppd.Solver(L0, 1, precision=prec, eta=1.0, L1=L1)
        s.set_problem(om, np.zeros(M, complex), np.zeros(M, np.int32))
        P = nufft.Plan(om, L0, L1)
        x = rng.normal(size=(L0, L1))
        yv = rng.normal(size=M) + 1j * rng.normal(size=M)
        assert rel(op_forward(s, x, dt), nufft.phi(x, P)) <= tol, (L0, L1)
        assert rel(op_adjoint(s, yv, dt), nufft.phi_adjoint(yv, P)) <= tol, (L0, L1)
        s.close()
