"""Refinement of the sampled screen where bonds end in different rounds: the CTAs of
a bond that is done run ahead of those of a bond that goes on, so every CTA must
still leave the refinement after the same step.  Few samples make many rounds; the
same run many times over, alone and in a batch of instances with other round
limits, equals the oracle bit for bit, its evaluated entries (a column or a row
per step) included."""
import numpy as np
import pytest

from test_gpu_parity import assert_same
from test_gpu_sampled import run_sampled, tt  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu

CASES = [([150, 9, 12, 200, 30], 6, 8), ([40, 40, 40], 1, 3), ([17, 60, 5, 33], 9, 64)]


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("host_loop", [False, True])
def test_bonds_end_in_different_rounds(tt, case, host_loop):  # noqa: F811
    n, nl, rook = CASES[case]
    w = dict(n=n, gen={"kind": "hilbert"})
    g, rc, o, orc, ost = run_sampled(tt, w, 1e-9, 12, 4000, nl, rook, host_loop=host_loop)
    for _ in range(1 if host_loop else 25):
        assert rc == orc
        assert_same(g, o)
        st = g.stats()
        assert st["sweeps"] == ost["sweeps"] and st["entries_screened"] == ost["entries_screened"]
        g.run(1e-9)
        rc = g.sync(allow=(tt.OK, tt.NOT_CONVERGED))


def test_batch_of_other_round_limits(tt):  # noqa: F811
    runs = [run_sampled(tt, dict(n=n, gen={"kind": "hilbert"}), 1e-9, 12, 4000, nl, rook)
            for n, nl, rook in CASES]
    single = [[g.core(k) for k in range(1, g.d + 1)] for g, *_ in runs]
    gs = [g for g, *_ in runs]
    for _ in range(10):
        tt.run_batch(gs, 1e-9)
        for (g, rc, o, *_), cores in zip(runs, single):
            assert g.sync(allow=(tt.OK, tt.NOT_CONVERGED)) == rc
            assert_same(g, o)
            for k in range(1, g.d + 1):
                np.testing.assert_array_equal(g.core(k), cores[k - 1])
