"""The sampled error with its middle cores on the tensor cores (split
integers, sorted samples), at the edges of its tiles: ranks around multiples
of 8 and 16, ranks past one accumulation (128), modes of a few and of many
indices, one to four middle cores, tables whose last mode runs there.  The
reference evaluates the GPU's own cores at the same samples in extended
precision, with the oracle's entries and sample indices.

Tolerance: X~ is a product of d cores, each entry at most a few units, with a
relative error of a few times 2^-53 per core and term; the errors of the
samples enter the reported norm through ||X~ - X~_exact|| / ||X||, a few
hundred times 2^-53 at these d and ranks: 1e-13 absolute."""
import numpy as np
import pytest

import oracle
from paper_2407_11290_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2407_11290_gb300 import ttcross
    return ttcross


def reference_error(w, cores, ns, seed):
    o = oracle.Oracle(w["n"], w["gen"], 1)
    idx = oracle.sample_indices(w["n"], ns, seed)
    x = np.array([o.entry(i) for i in idx], np.longdouble)
    cores = [c.astype(np.longdouble) for c in cores]
    v = cores[0][0, idx[:, 0], :]
    for m in range(1, len(cores)):
        v = np.concatenate([np.einsum("sp,psq->sq", v[i:i + 512], cores[m][:, idx[i:i + 512, m], :])
                            for i in range(0, ns, 512)])
    return float(np.sqrt(((x - v[:, 0]) ** 2).sum() / (x ** 2).sum()))


@pytest.mark.parametrize("w,ranks", [
    (W.hilbert(3, 90), (8, 9)),                                   # one middle core
    (dict(n=[40, 300, 260, 30], gen={"kind": "hilbert"}), (16, 15, 7)),
    (dict(n=[50, 2, 2048, 50], gen={"kind": "hilbert"}), (1, 1, 1)),
    (dict(n=[300, 3, 7, 290], gen={"kind": "hilbert"}), (17, 16, 15)),
    (W.hilbert(5, 64), (7, 8, 16, 9)),                            # tables' last mode
    (W.hilbert(6, 100), (12, 15, 16, 17, 13)),                    # two middle cores
    (dict(n=[70, 65, 33, 40, 31, 65, 66], gen={"kind": "hilbert"}), (9, 13, 15, 16, 14, 8)),
    (W.maxwellian(3, 3, 24), None),                               # past one accumulation
])
def test_sampled_error_against_extended_precision(tt, w, ranks):
    ns, seed = 70001, 99
    if ranks is None:
        c = tt.TTCross(w["n"], w["gen"], max_rank=160, nsamples=ns, seed=seed, residual="stored")
        c.run(1e-4)
        c.sync()
        assert max(c.ranks()) > 128
    else:
        c = tt.TTCross(w["n"], w["gen"], max_rank=max(ranks), bond_max_rank=list(ranks),
                       nsamples=ns, seed=seed, residual="stored")
        c.run(0.0)
        c.sync()
        assert tuple(c.ranks()[1:-1]) == ranks
    st, cores = c.stats(), c.cores()
    assert max(np.abs(g).max() for g in cores) < 16  # what the tolerance rests on
    ref = reference_error(w, cores, ns, seed)
    assert abs(st["err"] - ref) <= 1e-13, (st["err"], ref)


def test_host_stepped_check_is_the_same(tt):
    w = W.hilbert(5, 100)
    errs = []
    for host_loop in (False, True):
        c = tt.TTCross(w["n"], w["gen"], max_rank=32, nsamples=200000, host_loop=host_loop)
        c.run(1e-8)
        c.sync()
        errs.append(c.stats()["err"])
    assert errs[0] == errs[1]
