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


@pytest.mark.parametrize("n,gen,eps,cap,form", [
    ([64] * 6, {"kind": "hilbert"}, 1e-8, 64, dict(residual="stored")),
    ([64] * 4, {"kind": "maxwellian", "dx": 2, "dv": 2, "a_rho": 0.5, "a_u": 0.3, "a_T": 0.2, "vmin": -8.0,
                "vmax": 8.0}, 1e-3, 96, dict()),
    ([256] * 6, {"kind": "hilbert"}, 0.0, 24, dict(screen_samples=20000)),
])
def test_instance_in_less_memory(tt, n, gen, eps, cap, form):
    """Where its full memory is not free an instance does without what only makes runs
    faster, and returns the same: pivots and cores bit for bit, the error within
    the sampled error's tolerance (its middle cores run in FP64 then)."""
    import torch
    ok = (tt.OK, tt.NOT_CONVERGED)
    used(tt, [8] * 3, gen if gen["kind"] == "hilbert" else {"kind": "hilbert"}, max_rank=4, nsamples=100)[0].close()
    a, full = used(tt, n, gen, max_rank=cap, nsamples=300000, **form)
    a.run(eps)
    rc = a.sync(allow=ok)
    want = [a.core(k) for k in range(1, a.d + 1)], a.stats()["err"]
    a.close()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    room = full - max(8 << 20, full // 40)  # too little for all of it
    fill = torch.empty(free - room, dtype=torch.uint8, device="cuda")
    b, lean = used(tt, n, gen, max_rank=cap, nsamples=300000, **form)
    assert lean < full
    b.run(eps)
    assert b.sync(allow=ok) == rc
    for k in range(1, b.d + 1):
        assert (b.core(k) == want[0][k - 1]).all()
    assert abs(b.stats()["err"] - want[1]) <= 1e-12
    b.close()
    with pytest.raises(tt.TTCError) as e:  # a refusal leaves nothing behind
        tt.TTCross([512] * 6, {"kind": "hilbert"}, max_rank=64, residual="stored")
    assert e.value.status == tt.ERR_OOM
    del fill
    torch.cuda.empty_cache()
    c = tt.TTCross([12] * 3, {"kind": "hilbert"}, max_rank=8, nsamples=0)
    c.run(1e-6)
    assert c.sync() == tt.OK
