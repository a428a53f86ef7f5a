"""A sub-iteration that leaves a block as it is reads none of its data: with
every block skipped (active sets: the extra step of blocks that already have
a prox output) the launch takes less than half of a working step's time."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1701_01748_gb300 import ppd

pytestmark = pytest.mark.gpu


def subiter_us(s, n, masks=None):
    ppd.ppd_timing_enable(s.ctx, True)
    seen = (0.0, 0)
    for _ in range(2):   # the first call also warms up
        if masks is not None:
            ppd.ppd_set_active_sets(s.ctx, masks)
        s.iterate(n)
        ppd.ppd_timing_collect(s.ctx)
        last, seen = seen, ppd.ppd_timing_read(s.ctx)["subiter"]
    return (seen[0] - last[0]) / (seen[1] - last[1]) * 1e3


def test_skipped_blocks_are_not_read():
    L, M, d, n = 256, 4000000, 16, 10
    rng = np.random.default_rng(4)
    om = np.clip(rng.normal(0, 0.5, (M, 2)), -np.pi, np.nextafter(np.pi, 0))
    block = np.minimum(np.hypot(*om.T) * 8, d - 1).astype(np.int32)
    y = rng.normal(size=M) + 1j * rng.normal(size=M)
    t = {}
    for name, n_itr, masks in (("works", 2, None), ("skips", 1, np.ones((n, d), np.uint8))):
        s = ppd.Solver(L, d, eta=1e-9, n_itr=n_itr).set_problem(om, y, block)
        if masks is not None:   # every block active once: none is new afterwards
            ppd.ppd_set_active_sets(s.ctx, masks)
        s.iterate(n)
        t[name] = subiter_us(s, n, masks)
        s.close()
    assert t["skips"] < 0.5 * t["works"], t
