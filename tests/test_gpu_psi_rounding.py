"""Rounding of the synthesis against 64 bits, of clipped random coefficients:
1.18e-7 of the image's norm with the low and the high half of every pass summed
apart, 1.24e-7 in one accumulator, whose every addition rounds at the size of
the whole sum (64^2 to 2048^2, the same to 1 %).  The bound is between them."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from oracle import sara
from paper_1701_01748_gb300 import ppd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L0,L1", [(256, 256), (128, 512)])
def test_synthesis_error_against_64_bits(L0, L1):
    kappa, err = 1e-4, []
    s = ppd.Solver(L0, 1, L1=L1)
    for seed in range(4):
        c = np.clip(2 * kappa * np.random.default_rng(seed).standard_normal((9, L0, L1)), -kappa, kappa).astype(np.float32)
        cd, out = torch.from_numpy(c).cuda(), torch.empty(L0, L1, device="cuda")
        ppd.ppd_psi_synthesis(s.ctx, cd.data_ptr(), out.data_ptr(), torch.cuda.current_stream().cuda_stream)
        ref = sara.psi(c.astype(np.float64))
        err.append(np.linalg.norm(out.cpu().double().numpy() - ref) / np.linalg.norm(ref))
    s.close()
    assert np.mean(err) <= 1.21e-7
