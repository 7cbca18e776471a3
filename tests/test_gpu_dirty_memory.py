"""Instances whose memory held other data: what creation does not clear (the error check's
workspace and sample orders, step vectors, tile states, refinement lists) is written
before it is read.  The device is filled with NaN bit patterns and given back right
before the instance is made; FP64 pivots and cores equal the oracle's bit for bit,
every form's reported error is that of its cores at the oracle's sample indices
(1e-12 absolute, the tolerance of the sampled error) and no unwritten slot is read."""
import os

import numpy as np
import pytest

import oracle
from paper_2407_11290_gb300 import workloads as W

from test_gpu_parity import assert_same

pytestmark = pytest.mark.gpu

NS = 70000  # enough for the sorted samples


def dirty():
    import torch
    x = torch.full((1 << 29,), -1, dtype=torch.int32, device="cuda")  # 2 GB of 0xFF
    torch.cuda.synchronize()
    del x
    torch.cuda.empty_cache()


@pytest.mark.parametrize("w,eps,cap", [
    (dict(n=[40, 70, 66, 35], gen={"kind": "hilbert"}), 1e-9, 24),
    (W.maxwellian(2, 2, [24, 20, 33, 30]), 1e-4, 40),
    (dict(n=[30] * 6, gen={"kind": "hilbert"}), 1e-6, 16),
])
@pytest.mark.parametrize("form", [dict(), dict(residual="stored"), dict(precision="split"),
                                  dict(residual="stored", precision="split"), dict(screen_samples=2000)])
def test_uncleared_memory_is_not_read(w, eps, cap, form):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2407_11290_gb300 import ttcross as tt
    n, d = w["n"], len(w["n"])
    dirty()
    g = tt.TTCross(n, w["gen"], max_rank=cap, nsamples=NS, **form)
    g.run(eps, subtensor_grid=[2] * d)
    rc = g.sync(allow=(tt.OK, tt.NOT_CONVERGED))
    if form.get("precision") is None:
        o = oracle.Oracle(n, w["gen"], cap, nthreads=os.cpu_count() or 1, stored="residual" in form)
        if "screen_samples" in form:
            o.set_sampled(2000)
        assert o.run(eps, nsamples=NS)[0] == rc
        if w["gen"]["kind"] == "hilbert":
            assert_same(g, o)
        else:
            assert list(g.ranks()[1:-1]) == list(o.ranks())
    assert g.stats()["unscreened_slots"] == 0
    idx = oracle.sample_indices(n, NS)
    ref = oracle.Oracle(n, w["gen"], 1)
    x = np.array([ref.entry(i) for i in idx])
    cores = g.cores()
    v = cores[0][0, idx[:, 0], :]
    for m in range(1, d):
        v = np.concatenate([np.einsum("sp,psq->sq", v[i:i + 4096], cores[m][:, idx[i:i + 4096, m], :])
                            for i in range(0, NS, 4096)])
    err = float(np.sqrt(((x - v[:, 0]) ** 2).sum() / (x ** 2).sum()))
    assert abs(g.stats()["err"] - err) <= 1e-12, (g.stats()["err"], err)
    g.close()
