"""Gridding work items that hold several blocks of a tile: random block ids
(every tile mixes all blocks), item sizes below a group, not a multiple of it,
and larger than a tile's visibilities, both tile sides.  Operators against the
FP64 oracle (1e-5 FP32, 1e-10 FP64), four iterations with two inner steps
against the oracle's (1e-4, 1e-8: the tolerances of the trajectory tests)."""
from __future__ import annotations

import math

import numpy as np
import pytest
import torch

from oracle import nufft, ppd as oppd
from paper_1701_01748_gb300 import ppd

pytestmark = pytest.mark.gpu

F32, F64 = ppd.PPD_FP32_FP64NORMS, ppd.PPD_FP64_PLAIN


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("prec", [F32, F64])
@pytest.mark.parametrize("tile,chunk,blocks", [(16, 7, 5), (16, 100, 5), (16, 1024, 40), (32, 33, 5), (32, 0, 1)])
def test_items_of_several_blocks(prec, tile, chunk, blocks):
    L, M = 48, 6000
    rng = np.random.default_rng(blocks + chunk)
    om = np.clip(rng.normal(0, 0.2 * math.pi, (M, 2)), -math.pi, math.pi)
    block = rng.integers(0, blocks, M).astype(np.int32)
    y = rng.normal(size=M) + 1j * rng.normal(size=M)
    theta = rng.uniform(0.5, 2.0, M)
    S = oppd.make_setup(om, y, theta, block, blocks, L, eta=1e-6, n_itr=2)
    s = ppd.Solver(L, blocks, precision=prec, eta=1e-6, n_itr=2, tile=tile, chunk=chunk)
    s.set_problem(om, y, block, theta=theta)
    tol, itol, dt = (1e-5, 1e-4, torch.float32) if prec == F32 else (1e-10, 1e-8, torch.float64)
    st = torch.cuda.current_stream().cuda_stream
    yd = torch.tensor(np.stack([y.real, y.imag], 1), dtype=dt, device="cuda")
    ref = nufft.phi_adjoint(y, S.P)
    out = torch.empty((L, L), dtype=dt, device="cuda")
    ppd.ppd_op_adjoint(s.ctx, yd.data_ptr(), out.data_ptr(), st)
    assert rel(out.cpu().double().numpy(), ref) <= tol
    E = s.params()["tile"] + 8
    if s.params()["n_chunks"] * E * E * (8 if prec == F32 else 16) <= 32 << 20:
        out2 = torch.empty((L, L), dtype=dt, device="cuda")
        ppd.ppd_op_adjoint_noalloc(s.ctx, yd.data_ptr(), out2.data_ptr(), st)
        assert torch.equal(out, out2)
    x = rng.normal(size=(L, L))
    xd = torch.tensor(x, dtype=dt, device="cuda")
    ppd.ppd_op_forward(s.ctx, xd.data_ptr(), yd.data_ptr(), st)
    assert rel(yd.cpu().double().numpy() @ np.array([1.0, 1j]), nufft.phi(x, S.P)) <= tol
    state = oppd.init_state(S)
    for _ in range(4):
        oppd.iterate(state, S)
    s.iterate(4)
    assert rel(s.image(), state.x) <= itol
    s.close()
