"""ttcross_sampled_error_noalloc on cores with rows of zeros that meet large columns
(zero-padded ranks, a subspace expansion [U Z] against [V; 0]): the column, of
entries up to 2^300, contributes nothing, wherever its bond lies.  The reference is the
error of the same cores without those rows and columns.

Tolerance: the two TTs are the same tensor, and Gaussian cores of up to 32 terms keep a
chain of 5 cores within 6 * 32 * 2^-53 = 2.2e-14 of the norm of X~, the error
within less than that relative to itself: 1e-13, as between two evaluations."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("top", [30, 80, 300])
@pytest.mark.parametrize("n,s,bond", [
    ([20, 30, 40], [4, 9], 1),
    ([20, 30, 40], [4, 9], 2),               # the last core has the row
    ([64, 33, 64, 48, 64], [9, 16, 15, 7], 1),
    ([64, 33, 64, 48, 64], [9, 16, 15, 7], 3),
    ([64, 33, 64, 48, 64], [17, 32, 31, 16], 2),
])
def test_zero_rows(n, s, bond, top):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2407_11290_gb300 import ttcross
    rng = np.random.default_rng(sum(n) + sum(s) + top)
    sz = [1] + s + [1]
    cores = [rng.standard_normal((sz[m], n[m], sz[m + 1])) / np.sqrt(sz[m]) for m in range(len(n))]
    gone = [0, s[bond - 1] - 1]
    cores[bond - 1][:, :, gone] *= 2.0 ** top
    cores[bond][gone] = 0.0
    lean = list(cores)
    lean[bond - 1] = np.ascontiguousarray(np.delete(cores[bond - 1], gone, axis=2))
    lean[bond] = np.ascontiguousarray(np.delete(cores[bond], gone, axis=0))
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    got = []
    for cs in (lean, cores):
        ttcross.sampled_error_noalloc(n, {"kind": "hilbert"},
                                      [torch.from_numpy(c).cuda() for c in cs], 20000, 5, out)
        got.append(out.item())
    assert abs(got[1] - got[0]) <= 1e-13 * got[0], got
