"""Entries of a TT-cores tensor at the edge of the shared prefix vectors (core
ranks of 16, and of 17 where every entry runs from mode 0): ragged modes, both
residual forms and the float-float recompute screen.  Pivots and cores equal
the oracle's bit for bit."""
import os

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


@pytest.mark.parametrize("ranks", [[1, 9, 16, 5, 1], [1, 9, 17, 5, 1], [1, 1, 2, 2, 1]])
@pytest.mark.parametrize("residual,precision", [("recompute", "fp64"), ("stored", "fp64"),
                                                ("recompute", "split")])
def test_tt_entries_equal_oracle(tt, ranks, residual, precision):
    w = W.random_tt([33, 17, 65, 9], ranks, seed=5)
    g = tt.TTCross(w["n"], w["gen"], max_rank=20, nsamples=5000, residual=residual,
                   precision=precision)
    g.run(1e-11)
    rc = g.sync(allow=(tt.OK, tt.NOT_CONVERGED))
    o = oracle.Oracle(w["n"], w["gen"], 20, nthreads=os.cpu_count() or 1,
                      stored=residual == "stored")
    orc, _ = o.run(1e-11, nsamples=5000)
    assert rc == orc
    assert_same(g, o)
