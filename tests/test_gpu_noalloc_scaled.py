"""ttcross_sampled_error_noalloc on cores whose bonds are scaled: column k of a core
times 2^e, row k of the next times 2^-e, e up to 300, leaves the tensor as it was.

Tolerance: powers of two are exact, so the scaled cores keep the rounding bounds of
the unscaled ones: a chain of 5 cores of up to 32 terms is off by less than
6 * 32 * 2^-53 = 2.2e-14 of the norm of X~, the error by less than that relative to
itself (X~ is as large as X - X~ or smaller): 1e-13, as between two evaluations."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("top", [1, 30, 300])
@pytest.mark.parametrize("n,s", [
    ([20, 30, 40], [4, 9]),
    ([64, 33, 64, 48, 64], [9, 16, 15, 7]),
    ([64, 33, 64, 48, 64], [17, 32, 31, 16]),
])
def test_scaled_bonds(n, s, top):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2407_11290_gb300 import ttcross
    rng = np.random.default_rng(sum(n) + sum(s) + top)
    sz = [1] + s + [1]
    cores = [rng.standard_normal((sz[m], n[m], sz[m + 1])) / np.sqrt(sz[m]) for m in range(len(n))]
    cores[1][0] = 0.0  # a row of zeros
    scaled = [c.copy() for c in cores]
    for b in range(1, len(n)):
        e = rng.integers(-top, top + 1, sz[b])
        scaled[b - 1] = np.ldexp(scaled[b - 1], e[None, None, :])
        scaled[b] = np.ldexp(scaled[b], -e[:, None, None])
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    got = []
    for cs in (cores, scaled):
        ttcross.sampled_error_noalloc(n, {"kind": "hilbert"},
                                      [torch.from_numpy(c).cuda() for c in cs], 20000, 5, out)
        got.append(out.item())
    assert abs(got[1] - got[0]) <= 1e-13 * got[0], got
