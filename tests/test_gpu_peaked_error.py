"""The error of a cross of a tensor with one entry far above the rest: the cross finds
the peak (it starts there), no error sample holds it, and T has a column of 2^-t
against rows of R of 2^t.  The reported error equals that of the returned cores,
evaluated at the oracle's sample indices in extended precision.

Tolerance: the ranks are kept below the tensor's, so the error is far above the
roundings; X~ sums up to 16 terms a core, each within 2^-53 of terms that are up to
about a hundred times X, over 5 cores: 5 * 16 * 100 * 2^-53 = 9e-13 of rms(X),
1e-7 of errors of 1e-5 and more."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

NS = 10**5


@pytest.mark.parametrize("t", [0, 30, 60])
@pytest.mark.parametrize("n,cap,residual", [([32] * 6, 14, "recompute"), ([40, 50, 60, 41], 16, "stored"),
                                            ([200, 230, 210], 16, "recompute")])
def test_peaked_tensor(n, cap, residual, t):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2407_11290_gb300 import ttcross
    d, r = len(n), 25
    rng = np.random.default_rng(d)
    # a smooth part: sum_j 0.6^j prod_m cos(2 pi (k_j i_m / n_m + phase)) of other frequencies
    cores = []
    for m in range(d):
        c = np.zeros((1 if m == 0 else r, n[m], 1 if m == d - 1 else r))
        for j in range(r - 1):
            f = np.cos(2 * np.pi * (0.4 * (j + 1) * np.arange(n[m]) / n[m] + rng.random()))
            c[0 if m == 0 else j, :, 0 if m == d - 1 else j] = f * (0.6 ** j if m == 0 else 1.0)
        c[0 if m == 0 else r - 1, 0, 0 if m == d - 1 else r - 1] = 2.0 ** t if m == 0 else 1.0
        cores.append(c)
    seed = next(s for s in range(1, 99)
                if not (oracle.sample_indices(n, NS, s).sum(axis=1) == 0).any())
    c = ttcross.TTCross(n, {"kind": "tt", "ranks": [1] + [r] * (d - 1) + [1], "cores": cores}, max_rank=cap,
                        nsamples=NS, seed=seed, residual=residual)
    c.run(0.0)
    c.sync()
    idx = oracle.sample_indices(n, NS, seed)

    def values(cs):
        v = cs[0].astype(np.longdouble)[0, idx[:, 0], :]
        for m in range(1, d):
            g = cs[m].astype(np.longdouble)
            v = np.concatenate([np.einsum("sp,psq->sq", v[i:i + 1024], g[:, idx[i:i + 1024, m], :])
                                for i in range(0, NS, 1024)])
        return v[:, 0]

    x = values(cores)
    ref = float(np.sqrt(((x - values([c.core(k) for k in range(1, d + 1)])) ** 2).sum() / (x ** 2).sum()))
    got = c.stats()["err"]
    assert ref > 1e-5 and abs(got - ref) <= 1e-7 * ref, (got, ref)
