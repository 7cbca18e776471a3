"""Cores rebuilt from the pivots (eight rows a warp up to 64 pivots, one above;
the pivot rows' history in shared or in device memory): ranks on both sides of
the line, row counts that leave a remainder of a group, equal to the sweeps'
cores bit for bit."""
import numpy as np
import pytest

from paper_2407_11290_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ranks,cap", [
    ([5, 7], [1, 1, 1], 4),
    ([9, 9, 10, 9], [1, 9, 64, 9, 1], 72),
    ([9, 9, 10, 9], [1, 9, 65, 9, 1], 72),
    ([13, 12, 11, 13], [1, 13, 130, 13, 1], 140),
])
def test_rebuilt_cores_equal_the_sweeps(n, ranks, cap):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2407_11290_gb300 import ttcross as tt
    w = W.random_tt(n, ranks, seed=5)
    g = tt.TTCross(w["n"], w["gen"], max_rank=cap, nsamples=0)
    g.run(1e-11)
    g.sync(allow=(tt.OK, tt.NOT_CONVERGED))
    ref = g.cores()
    g.rebuild_cores()
    for a, b in zip(g.cores(), ref):
        np.testing.assert_array_equal(a, b)
