"""Kaiser-Bessel weights of the visibility kernels: Phi and Phi^dagger against
the FP64 oracle at coordinates where a tap's weight polynomial ends (on grid
points, one ulp beside them, half-way, the ends of the band), for the default
shape (polynomials) and for shapes whose FP64 weights come from the Bessel
function.  Tolerances: those of the operator tests (1e-5 in FP32, whose
polynomials serve the default shape; 1e-10 in FP64)."""
from __future__ import annotations

import math

import numpy as np
import pytest

from oracle import nufft
from paper_1701_01748_gb300 import ppd
from test_gpu_parity import op_adjoint, op_forward, rel

pytestmark = pytest.mark.gpu

F32, F64 = ppd.PPD_FP32_FP64NORMS, ppd.PPD_FP64_PLAIN


@pytest.mark.parametrize("prec,beta", [(F32, 0.0), (F64, 0.0), (F64, 10.0), (F64, 18.0), (F64, 40.0), (F64, 90.0)])
def test_weights_at_the_ends_of_a_tap(prec, beta):
    L, K = 32, 64
    cells = np.arange(-K // 2, K // 2) * (2 * math.pi / K)
    edge = np.concatenate([cells, np.nextafter(cells, 4), np.nextafter(cells, -4), cells + math.pi / K])
    edge = np.clip(edge, -math.pi, np.nextafter(math.pi, 0))
    rng = np.random.default_rng(8)
    om = np.concatenate([np.stack([edge, rng.permutation(edge)], 1), rng.uniform(-math.pi, math.pi, (500, 2))])
    M = om.shape[0]
    s = ppd.Solver(L, 1, precision=prec, eta=1.0, kb_beta=beta)
    s.set_problem(om, np.zeros(M, complex), np.zeros(M, np.int32))
    P = nufft.Plan(om, L, beta=beta if beta > 0 else None)
    tol = 1e-5 if prec == F32 else 1e-10
    x = rng.random((L, L))
    assert rel(op_forward(s, x, prec), nufft.phi(x, P)) <= tol
    yv = rng.normal(size=M) + 1j * rng.normal(size=M)
    assert rel(op_adjoint(s, yv, prec), nufft.phi_adjoint(yv, P)) <= tol
    s.close()
