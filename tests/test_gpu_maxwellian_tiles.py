"""Maxwellian entries formed from a tile's row and column data: position /
velocity splits in every place of the bond (also one position or one velocity
mode, and more modes than the tiles' tables hold), ragged tiles.  Entries come
from CUDA's exp against glibc's, so pivots are compared with the near-tie
re-sync of ``replay_with_resync``."""
import pytest

from paper_2407_11290_gb300 import workloads as W

from test_gpu_parity import replay_with_resync

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2407_11290_gb300 import ttcross
    return ttcross


@pytest.mark.parametrize("w", [
    W.maxwellian(1, 1, [40, 33]), W.maxwellian(1, 3, [9, 70, 12, 11]),
    W.maxwellian(3, 1, [9, 8, 11, 65]), W.maxwellian(2, 1, [37, 10, 66]),
    W.maxwellian(4, 5, [3, 4, 3, 2, 5, 4, 6, 5, 3]),
    W.maxwellian_xv(1, 50, 35), W.maxwellian_xv(2, 13, 17), W.maxwellian_xv(5, 3, 4),
])
@pytest.mark.parametrize("stored", [False, True])
def test_maxwellian_tiles(tt, w, stored):
    kw = dict(max_rank=6, nsamples=3000, residual="stored" if stored else "recompute")
    g = tt.TTCross(w["n"], w["gen"], **kw)
    g.run(1e-3)
    g.sync(allow=(tt.OK, tt.NOT_CONVERGED))
    replay_with_resync(g, w, 1e-3, 6, 3000, rel=1e-12, stored=stored, first_stage=True)
