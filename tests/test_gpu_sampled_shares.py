"""The sampled screen and its refinement steps share a bond among a part of the
grid's CTAs: fewer CTAs than bonds (all of them take every bond), as many, a
remainder, and columns long enough that all CTAs share each of them, equal to
the oracle bit for bit."""
import numpy as np
import pytest

from paper_2407_11290_gb300 import workloads as W

from test_gpu_parity import assert_same
from test_gpu_sampled import run_sampled, tt  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,cap,ctas", [
    ([9, 12, 10, 11, 8], 12, 1),
    ([9, 12, 10, 11, 8], 12, 4),
    ([9, 12, 10, 11, 8], 12, 7),
    ([2100, 30, 2500], 14, 2),   # rows past 16 passes of a one-CTA share
    ([40, 1500, 41], 16, 5),     # past them as the ranks grow
])
@pytest.mark.parametrize("host_loop", [False, True])
def test_shares_of_the_grid(tt, n, cap, ctas, host_loop):  # noqa: F811
    w = dict(n=n, gen={"kind": "hilbert"})
    g, rc, o, orc, ost = run_sampled(tt, w, 1e-10, cap, 3000, 300, 5, grid_ctas=ctas,
                                     host_loop=host_loop)
    assert rc == orc
    assert_same(g, o)
    st = g.stats()
    assert st["sweeps"] == ost["sweeps"] and st["entries_screened"] == ost["entries_screened"]
    assert np.isfinite(st["err"])
