"""FP64 weights on both sides of the rule that takes the polynomials (fit
error up to 1e-15: shapes up to beta = 28) or the Bessel function.  At beta =
90 the polynomials would be off by 8e-12 at most, 1.6e-12 rms, in weights up to 1; the
Bessel function, here and in the oracle, is off by 90 x 2^-53 = 1e-14 through
its argument.  The tolerance is ten times that."""
from __future__ import annotations

import math

import numpy as np
import pytest

from oracle import nufft
from paper_1701_01748_gb300 import ppd
from test_gpu_parity import op_adjoint, op_forward, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("beta", [0.0, 28.0, 30.0, 90.0])
def test_fp64_weights_at_the_rule(beta):
    L, M = 32, 3000
    rng = np.random.default_rng(9)
    om = rng.uniform(-math.pi, math.pi, (M, 2))
    s = ppd.Solver(L, 1, precision=ppd.PPD_FP64_PLAIN, eta=1.0, kb_beta=beta)
    s.set_problem(om, np.zeros(M, complex), np.zeros(M, np.int32))
    P = nufft.Plan(om, L, beta=beta if beta > 0 else None)
    x = rng.random((L, L))
    assert rel(op_forward(s, x, ppd.PPD_FP64_PLAIN), nufft.phi(x, P)) <= 1e-13
    yv = rng.normal(size=M) + 1j * rng.normal(size=M)
    assert rel(op_adjoint(s, yv, ppd.PPD_FP64_PLAIN), nufft.phi_adjoint(yv, P)) <= 1e-13
    s.close()
