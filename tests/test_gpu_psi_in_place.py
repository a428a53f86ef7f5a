"""Psi^dagger with the image in the coefficients' own Dirac part, which every
basis reads and the result replaces: the same coefficients as from a separate
image, bit for bit; Psi into the Dirac part likewise."""
from __future__ import annotations

import pytest
import torch

from paper_1701_01748_gb300 import ppd

pytestmark = pytest.mark.gpu

F32, F64 = ppd.PPD_FP32_FP64NORMS, ppd.PPD_FP64_PLAIN


@pytest.mark.parametrize("prec", [F32, F64])
@pytest.mark.parametrize("L0,L1", [(16, 16), (48, 80), (256, 256), (720, 640)])
def test_image_in_the_dirac_part(prec, L0, L1):
    s = ppd.Solver(L0, 1, L1=L1, precision=prec)
    st = torch.cuda.current_stream().cuda_stream
    dt = torch.float32 if prec == F32 else torch.float64
    x = torch.randn(L0, L1, dtype=dt, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    want, c = torch.empty(9, L0, L1, dtype=dt, device="cuda"), torch.zeros(9, L0, L1, dtype=dt, device="cuda")
    ppd.ppd_psi_analysis(s.ctx, x.data_ptr(), want.data_ptr(), st)
    c[0] = x
    ppd.ppd_psi_analysis(s.ctx, c.data_ptr(), c.data_ptr(), st)
    assert torch.equal(c, want)
    back = torch.empty_like(x)
    ppd.ppd_psi_synthesis(s.ctx, want.data_ptr(), back.data_ptr(), st)
    ppd.ppd_psi_synthesis(s.ctx, c.data_ptr(), c.data_ptr(), st)
    assert torch.equal(c[0], back)
    s.close()
