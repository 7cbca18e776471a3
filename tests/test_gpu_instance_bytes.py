"""Device memory of an instance, from the free memory around its creation.  The mixed stored
form brings every carried tile up to date in every screen: it keeps no tile
states and no step history, which make up for its FP32 shadows of T and R (8.4 MB
here) against the FP64 form."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2407_11290_gb300 import ttcross
    return ttcross


def used(tt, *args, **kw):
    import torch
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    c = tt.TTCross(*args, **kw)
    torch.cuda.synchronize()
    got = before - torch.cuda.mem_get_info()[0]
    return c, got


def test_mixed_stored_form_keeps_no_lazy_state(tt):
    n, g = [64] * 4, {"kind": "hilbert"}
    used(tt, [8] * 3, g, max_rank=4, nsamples=100)[0].close()  # the context and the module
    a, fp64 = used(tt, n, g, max_rank=64, nsamples=1000, residual="stored")
    b, split = used(tt, n, g, max_rank=64, nsamples=1000, residual="stored", precision="split")
    assert split <= fp64 + (4 << 20), (split, fp64)  # (allocations come in pages of 2 MB)
