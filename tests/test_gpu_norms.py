"""Block norms of the FP32 path: FP64 precision and FP64 range over the lanes.

The first iteration from x = 0 has Phi xt = 0, so a block's residual is the
norm of its data.  The squares are formed in FP32 (a product and a fused
multiply-add, each within 2^-24), everything after them is summed to FP64
precision, so the norm is within 2^-24.

The whole iteration scales with the data and the bounds (and eta inversely),
exactly so for a power of two: at 2^62 every square is still a finite FP32
value (at most 14.6 * 2^124 = 3.1e38), the sum of a lane's few or of a warp's
is not.  What may differ from the small problem is where the sums are rounded,
in FP64 or with the FP32 compensation: below 1e-12."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1701_01748_gb300 import ppd

pytestmark = pytest.mark.gpu

L, BLOCKS = 64, 2


def data(M):
    rng = np.random.default_rng(M)
    om = np.clip(rng.normal(0, 0.8, (M, 2)), -np.pi, np.nextafter(np.pi, 0))
    y = np.clip(rng.normal(0, 1.5, (M, 2)), -2.7, 2.7).astype(np.float32).astype(np.float64) @ np.array([1, 1j])
    block = rng.integers(0, BLOCKS, M).astype(np.int32)
    return om, y, block, rng.uniform(0.5, 1.0, M)


# one group per warp, and shares of about 34 groups (runs that go on over groups)
@pytest.mark.parametrize("M", [3000, 4000000])
@pytest.mark.parametrize("cfg", [dict(n_itr=1), dict(n_itr=3, inner_tol=1e-3), dict(n_itr=3, inner_solver=1)])
def test_norms_keep_fp64_precision_and_range(M, cfg):
    om, y, block, U = data(M)
    ref = np.sqrt(np.bincount(block, np.abs(y) ** 2, BLOCKS))
    got = []
    for k in (0, 62):
        s = ppd.Solver(L, BLOCKS, eta=1e-4 / M * 2.0 ** -k, **cfg)
        s.set_problem(om, y * 2.0 ** k, block, U=U, eps=0.3 * ref * 2.0 ** k)
        st = s.iterate(1)
        got.append((st["block_residual"] * 2.0 ** -k, st["inner_steps"], s.image()))
        s.close()
    for res, _, _ in got:
        assert np.abs(res / ref - 1).max() <= 2.0 ** -24
    assert np.abs(got[1][0] / got[0][0] - 1).max() <= 1e-10
    assert np.array_equal(got[0][1], got[1][1])
    assert np.linalg.norm(got[1][2] - got[0][2]) <= 1e-6 * np.linalg.norm(got[0][2])
