"""ttcross_sampled_error_noalloc over core sizes and mode sizes at the edges of
its two forms: the split-integer products (core sizes up to 32 in tiles of 8 and
16, middle modes up to 256, at least 16384 samples) and the FP64 warp chains
beyond.  The reference evaluates the same cores at the oracle's sample indices
(every index where the samples are as many as the entries) in extended
precision.

Tolerance: Gaussian cores give X~ of the size of its terms' norm, so a chain of
d cores of up to 40 terms is off by less than 6 * 40 * 2^-53 = 3e-14 of the
norm of X~, and the reported error by less than that relative to itself (X~ is
as large as X - X~ or smaller): 1e-13."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2407_11290_gb300 import ttcross
    return ttcross


@pytest.mark.parametrize("n,s,ns", [
    ([30, 256, 40], [8, 9], 16384),
    ([30, 257, 40], [8, 9], 20000),            # a middle mode past the tiles' keys
    ([200, 5, 1, 70], [16, 15, 7], 70001),
    ([64, 64, 64, 64, 64], [17, 32, 31, 16], 16385),
    ([64, 64, 64, 64, 64], [17, 33, 31, 16], 16385),  # a core past 32
    ([9, 100, 33, 2, 65, 11], [1, 24, 25, 8, 1], 50000),
    ([40, 40, 40], [3, 2], 16383),             # too few samples for the tiles
])
def test_noalloc_against_extended_precision(tt, n, s, ns):
    import torch
    rng = np.random.default_rng(sum(n) + sum(s))
    sz = [1] + s + [1]
    cores = [rng.standard_normal((sz[m], n[m], sz[m + 1])) / np.sqrt(sz[m]) for m in range(len(n))]
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    got = []
    for _ in range(2):
        tt.sampled_error_noalloc(n, {"kind": "hilbert"}, [torch.from_numpy(c).cuda() for c in cores],
                                 ns, 5, out)
        got.append(out.item())
    assert got[0] == got[1]
    if ns >= np.prod(n):  # then the error runs over every entry
        idx = np.stack(np.unravel_index(np.arange(np.prod(n)), n, order="F"), axis=1)
    else:
        idx = oracle.sample_indices(n, ns, 5)
    x = (1.0 / (1.0 + idx.sum(axis=1))).astype(np.longdouble)
    v = cores[0].astype(np.longdouble)[0, idx[:, 0], :]
    for m in range(1, len(n)):
        c = cores[m].astype(np.longdouble)
        v = np.concatenate([np.einsum("sp,psq->sq", v[i:i + 1024], c[:, idx[i:i + 1024, m], :])
                            for i in range(0, len(idx), 1024)])
    ref = float(np.sqrt(((x - v[:, 0]) ** 2).sum() / (x ** 2).sum()))
    assert abs(got[0] - ref) <= 1e-13 * ref, (got[0], ref)


def test_noalloc_nonfinite_core(tt):
    import torch
    n, sz = [20, 30, 20], [1, 4, 4, 1]
    for bad in (float("inf"), float("nan")):
        cores = [torch.ones(sz[m], n[m], sz[m + 1], dtype=torch.float64, device="cuda")
                 for m in range(3)]
        cores[1][2, 7, 1] = bad
        out = torch.zeros(1, dtype=torch.float64, device="cuda")
        tt.sampled_error_noalloc(n, {"kind": "hilbert"}, cores, 11000, 5, out)   # FP64 chains
        a = out.item()
        tt.sampled_error_noalloc([20, 30, 40], {"kind": "hilbert"},
                                 cores[:2] + [torch.ones(4, 40, 1, dtype=torch.float64, device="cuda")],
                                 20000, 5, out)
        assert not np.isfinite(a) and not np.isfinite(out.item())
