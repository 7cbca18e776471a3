"""ttcross_sampled_error_noalloc past the sample counts (4096 slots of one batch: 4,194,304
samples at core sizes up to 16, 2,097,152 up to 32) where a slot takes several
batches of samples one after the other, with a ragged last batch; a peak that some
samples hit sends part of every batch to the FP64 chains.  The reference is the FP64
form, reached by padding one bond with zeros to size 33.

Tolerance: positive cores of up to 32 terms keep both forms within
3 * 33 * 2^-53 = 1.1e-14 of X~, the errors within 1e-13 of each other."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s,ns", [(9, 4194304 + 2 * 1024 + 5), (16, 2 * 4194304 + 1), (17, 2097152 + 777),
                                  (32, 2097152)])
def test_slots_of_several_batches(s, ns):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2407_11290_gb300 import ttcross
    n = [256, 255, 250]
    rng = np.random.default_rng(s)
    cores = [0.5 + rng.random((1, n[0], s)), 0.5 + rng.random((s, n[1], s)), 0.5 + rng.random((s, n[2], 1))]
    for c in cores:  # the last term is 2^50 at one entry
        c[-1, :, -1] = 0.0
    cores[0][0, :, -1] = 0.0
    cores[0][0, 7, -1] = cores[1][-1, 8, -1] = 1.0
    cores[2][-1, 9, 0] = 2.0 ** 50
    wide = [np.pad(cores[0], ((0, 0), (0, 0), (0, 33 - s))), np.pad(cores[1], ((0, 33 - s), (0, 0), (0, 0))),
            cores[2]]
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    got = []
    for cs in (cores, wide):
        ttcross.sampled_error_noalloc(n, {"kind": "hilbert"}, [torch.from_numpy(c).cuda() for c in cs], ns, 3,
                                      out)
        got.append(out.item())
    assert abs(got[0] - got[1]) <= 1e-13 * got[1], got
