"""ttc_stats of stored runs whose every screen brings every carried entry up to date
(ranks prescribed, so each bond takes a pivot in each decision): 8 bytes written
per fresh entry, 8 read and 8 written per carried one, an FMA per carried one and
r_k per fresh one, wherever the tile edges lie and with pieces."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "split"])
@pytest.mark.parametrize("edge,grid", [(0, None), (32, None), (64, [2, 3, 1])])
def test_stored_bytes_of_eager_screens(precision, edge, grid):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2407_11290_gb300 import ttcross as tt
    n, cap = [37, 145, 69], 6
    g = tt.TTCross(n, {"kind": "hilbert"}, max_rank=cap, nsamples=5000, residual="stored", precision=precision)
    g.set_plan(edge, 0)
    g.run(0.0, subtensor_grid=grid)
    g.sync()
    st = g.stats()
    assert list(g.ranks()) == [1, cap, cap, 1]
    fresh = kept = fmas = 0
    old = [0, 0]
    for r in range(1, st["sweeps"] + 1):
        size = [n[0] * n[1] * r, r * n[1] * n[2]]
        for b in range(2):
            fresh += size[b] - old[b]
            kept += old[b]
            fmas += (size[b] - old[b]) * r + old[b]
        old = size
    assert (st["entries_fresh"], st["entries_screened"]) == (fresh, fresh + kept)
    assert st["stored_bytes"] == 8 * (fresh + 2 * kept)
    assert st["screen_fmas"] == fmas
