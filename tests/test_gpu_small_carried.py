"""Stored screens with few carried tiles, which CTAs take one at a time (an eighth of the rows
to a warp): superblocks of one tile, rows that leave warps without any, 32-wide
tiles, ragged pieces, and counts on both sides of the line (four tiles a CTA, reached with
few CTAs).  FP64 pivots, inverses and cores equal the oracle's bit for bit; the
mixed form's results do not depend on the number of CTAs, which decides how its tiles
are taken."""
import os

import numpy as np
import pytest

import oracle

from test_gpu_parity import assert_same

pytestmark = pytest.mark.gpu

CASES = [([13, 12], 1e-10, 13), ([65, 70, 3], 1e-9, 20), ([70, 69, 66], 1e-10, 30), ([9, 200, 7, 90], 1e-9, 20),
         ([2, 130, 2], 1e-6, 4)]


@pytest.fixture(scope="module")
def tt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2407_11290_gb300 import ttcross
    return ttcross


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("edge,pieces,ctas", [(0, 0, 0), (32, 0, 0), (64, 2, 0), (0, 0, 3), (32, 2, 5), (0, 0, 1)])
def test_few_carried_tiles(tt, case, edge, pieces, ctas):
    n, eps, cap = CASES[case]
    grid = [min(pieces, v) for v in n] if pieces else None
    ok = (tt.OK, tt.NOT_CONVERGED)
    g = tt.TTCross(n, {"kind": "hilbert"}, max_rank=cap, nsamples=3000, residual="stored", grid_ctas=ctas)
    g.set_plan(edge, 0)
    g.run(eps, subtensor_grid=grid)
    rc = g.sync(allow=ok)
    o = oracle.Oracle(n, {"kind": "hilbert"}, cap, nthreads=os.cpu_count() or 1, stored=True)
    assert rc == o.run(eps, nsamples=3000)[0]
    assert_same(g, o)
    for k in range(1, o.d):
        np.testing.assert_array_equal(g.pivot_inverse(k), o.U(k - 1))
    runs = []
    for c in (ctas, 0, 2):
        s = tt.TTCross(n, {"kind": "hilbert"}, max_rank=cap, nsamples=3000, residual="stored", precision="split",
                       grid_ctas=c)
        s.set_plan(edge, 0)
        s.run(eps, subtensor_grid=grid)
        s.sync(allow=ok)
        assert s.stats()["unscreened_slots"] == 0
        runs.append([s.core(k) for k in range(1, s.d + 1)])
    for other in runs[1:]:
        for a, b in zip(runs[0], other):
            np.testing.assert_array_equal(a, b)
