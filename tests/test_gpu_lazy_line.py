"""Stored residuals that grow past the size from which on carried tiles wait for their
steps (48 MB of E): the first sweeps bring every tile up to date, the later ones only
those that may hold the pivot, from the states that the eager sweeps left.  Tile
edges, ragged pieces, more pivots than a tile may have pending, a batch of
instances on both sides of the line: pivots, pivot inverses and cores equal the
oracle's bit for bit, and fewer bytes of E are moved than by eager screens alone."""
import os

import numpy as np
import pytest

import oracle
from paper_2407_11290_gb300 import workloads as W

from test_gpu_parity import assert_same

pytestmark = pytest.mark.gpu

BIG = [(dict(n=[40, 300, 310, 35], gen={"kind": "hilbert"}), 1e-9, 24),
       (W.random_tt([30, 141, 137, 30], [1, 30, 58, 30, 1], seed=9), 1e-11, 64)]
SMALL = dict(n=[40, 60, 41, 35], gen={"kind": "hilbert"}), 1e-9, 24


@pytest.fixture(scope="module")
def tt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2407_11290_gb300 import ttcross
    return ttcross


@pytest.fixture(scope="module")
def truth():
    out = []
    for w, eps, cap in BIG + [SMALL]:
        o = oracle.Oracle(w["n"], w["gen"], cap, nthreads=os.cpu_count() or 1, stored=True)
        out.append((o, o.run(eps, nsamples=20000)[0]))
    return out


def check(g, o, lazy):
    assert_same(g, o)
    for k in range(1, o.d):
        np.testing.assert_array_equal(g.pivot_inverse(k), o.U(k - 1))
    st = g.stats()
    carried = st["entries_screened"] - st["entries_fresh"]
    eager = 8 * (st["entries_fresh"] + 2 * carried)  # a read and a write of every carried entry
    assert not lazy or st["stored_bytes"] < 0.9 * eager


@pytest.mark.parametrize("case", range(2))
@pytest.mark.parametrize("edge,grid,host_loop", [(0, None, False), (32, None, False),
                                                 (64, [1, 2, 3, 2], False), (0, [3, 1, 5, 2], True)])
def test_runs_across_the_line(tt, truth, case, edge, grid, host_loop):
    w, eps, cap = BIG[case]
    o, orc = truth[case]
    g = tt.TTCross(w["n"], w["gen"], max_rank=cap, nsamples=20000, residual="stored", host_loop=host_loop)
    g.set_plan(edge, 0)
    g.run(eps, subtensor_grid=grid)
    assert g.sync(allow=(tt.OK, tt.NOT_CONVERGED)) == orc
    check(g, o, True)


def test_batch_on_both_sides_of_the_line(tt, truth):
    gs = [tt.TTCross(w["n"], w["gen"], max_rank=cap, nsamples=20000, residual="stored")
          for w, _, cap in BIG + [SMALL]]
    tt.run_batch(gs, [eps for _, eps, _ in BIG + [SMALL]])
    for i, (g, (o, orc)) in enumerate(zip(gs, truth)):
        assert g.sync(allow=(tt.OK, tt.NOT_CONVERGED)) == orc
        check(g, o, i < 2)
