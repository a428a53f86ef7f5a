"""SARA analysis and synthesis at the sizes where their tiling changes: levels
smaller than a tile, sides that are not multiples of the small or the large
tile, columns that wrap, levels whose rows are not 16-byte aligned, and device
pointers that are aligned to one value only.  Against the FP64 oracle, with
the tolerances of the operator tests (1e-5 in FP32, 1e-10 in FP64)."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from oracle import sara
from paper_1701_01748_gb300 import ppd

pytestmark = pytest.mark.gpu

F32, F64 = ppd.PPD_FP32_FP64NORMS, ppd.PPD_FP64_PLAIN


@pytest.mark.parametrize("prec,offset", [(F32, 0), (F32, 1), (F32, 2), (F64, 0), (F64, 1)])
@pytest.mark.parametrize("shape", [(16, 16), (16, 48), (64, 128), (80, 432), (240, 192), (640, 576)])
def test_tiles(shape, prec, offset):
    n0, n1 = shape
    dt = torch.float32 if prec == F32 else torch.float64
    tol = 1e-5 if prec == F32 else 1e-10
    rng = np.random.default_rng(n0 + n1)
    x, c = rng.normal(size=shape), rng.normal(size=(9,) + shape)

    def place(a):
        t = torch.zeros(a.size + offset, dtype=dt, device="cuda")
        t[offset:] = torch.tensor(a.ravel(), dtype=dt, device="cuda")
        return t[offset:]

    s = ppd.Solver(n0, 1, precision=prec, L1=n1)
    xd, cd, co, xo = place(x), place(c), place(np.zeros_like(c)), place(np.zeros_like(x))
    st = torch.cuda.current_stream().cuda_stream
    ppd.ppd_psi_analysis(s.ctx, xd.data_ptr(), co.data_ptr(), st)
    ppd.ppd_psi_synthesis(s.ctx, cd.data_ptr(), xo.data_ptr(), st)
    got_c, got_x = co.double().cpu().numpy().reshape(c.shape), xo.double().cpu().numpy().reshape(shape)
    ref_c, ref_x = sara.psi_adjoint(x), sara.psi(c)
    assert np.linalg.norm(got_c - ref_c) <= tol * np.linalg.norm(ref_c)
    assert np.linalg.norm(got_x - ref_x) <= tol * np.linalg.norm(ref_x)
    s.close()
