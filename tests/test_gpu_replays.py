"""Alg. 4 replays at the edges of their groups (eight rows a warp up to 64
pivots, one row a warp above) and of both dealings (a single run, whose replays
keep SMs of their own, and a batch): mode sizes around multiples of eight,
ranks across 64.  Pivots, pivot inverses and cores equal the oracle's bit for
bit; a batch equals its single runs."""
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


SHAPES = [([9, 17, 33, 9], [1, 9, 66, 9, 1]), ([8, 7, 1, 9, 8], [1, 8, 20, 20, 8, 1]),
          ([33, 2, 40, 5], [1, 33, 63, 5, 1]), ([5, 24, 25, 6], [1, 5, 65, 6, 1])]


def test_replay_groups_single_and_batch(tt):
    ws = [W.random_tt(n, r, seed=31 + i) for i, (n, r) in enumerate(SHAPES)]
    single, batch = [], []
    for w in ws:
        g = tt.TTCross(w["n"], w["gen"], max_rank=72, nsamples=0, residual="stored")
        g.run(1e-12)
        rc = g.sync(allow=(tt.OK, tt.NOT_CONVERGED))
        o = oracle.Oracle(w["n"], w["gen"], 72, nthreads=os.cpu_count() or 1, stored=True)
        orc, _ = o.run(1e-12, nsamples=0)
        assert rc == orc
        assert_same(g, o)
        for k in range(1, o.d):
            np.testing.assert_array_equal(g.pivot_inverse(k), o.U(k - 1))
        single.append(g)
        batch.append(tt.TTCross(w["n"], w["gen"], max_rank=72, nsamples=0, residual="stored"))
    tt.run_batch(batch, 1e-12)
    for a, b in zip(single, batch):
        b.sync(allow=(tt.OK, tt.NOT_CONVERGED))
        for x, y in zip(a.cores(), b.cores()):
            np.testing.assert_array_equal(x, y)
        for k in range(1, a.d):
            np.testing.assert_array_equal(a.pivot_inverse(k), b.pivot_inverse(k))
