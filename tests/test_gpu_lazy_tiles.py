"""The stored form's carried tiles, brought up to date only when a candidate may
lie in them: tile edges, subtensor grids with ragged pieces, superblocks whose
tiles straddle prefix blocks, enough pivots for tiles to wait longer than their
limit of pending steps, and refinements of the threshold (pivots appended without a
screen in between).  Pivots, pivot inverses and cores equal the oracle's bit
for bit, persistent and host-stepped."""
import os

import numpy as np
import pytest

import oracle
from paper_2407_11290_gb300 import workloads as W

from test_gpu_parity import assert_same

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2407_11290_gb300 import ttcross
    return ttcross


CASES = [
    (dict(n=[100, 70, 130, 65], gen={"kind": "hilbert"}), 1e-12, 30),
    (dict(n=[65, 64, 63, 33, 40], gen={"kind": "hilbert"}), 1e-9, 24),
    (W.random_tt([30, 41, 37, 30], [1, 30, 58, 30, 1], seed=9), 1e-11, 64),
    (dict(n=[9, 200, 7, 90], gen={"kind": "hilbert"}), 0.0, 9),
]


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("edge,grid,host_loop", [(0, None, False), (32, None, False),
                                                 (64, [1, 2, 1, 3, 2], False),
                                                 (0, [3, 1, 5, 2, 1], True)])
def test_lazy_tiles_equal_oracle(tt, case, edge, grid, host_loop):
    w, eps, cap = CASES[case]
    g = tt.TTCross(w["n"], w["gen"], max_rank=cap, nsamples=20000, residual="stored",
                   host_loop=host_loop)
    g.set_plan(edge, 0)
    g.run(eps, subtensor_grid=None if grid is None else grid[:len(w["n"])])
    rc = g.sync(allow=(tt.OK, tt.NOT_CONVERGED))
    o = oracle.Oracle(w["n"], w["gen"], cap, nthreads=os.cpu_count() or 1, stored=True)
    orc, _ = o.run(eps, nsamples=20000)
    assert rc == orc
    assert_same(g, o)
    for k in range(1, o.d):
        np.testing.assert_array_equal(g.pivot_inverse(k), o.U(k - 1))
