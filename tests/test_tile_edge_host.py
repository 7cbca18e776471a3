"""A stored run keeps the tile edge of its first plan (its tile states and candidate
lists are numbered by it), so 32-wide tiles, once taken, have to fit the candidate
slots at every later rank up to the caps: the stored form's slots hold four tiles
for each 64-wide one at the caps.  Replayed on the host (no GPU)."""
import numpy as np
import pytest

from paper_2407_11290_gb300 import ttcross


@pytest.mark.parametrize("seed", range(4))
def test_narrow_tiles_fit_the_stored_slots(seed):
    rng = np.random.default_rng(seed)
    for _ in range(60):
        d = int(rng.integers(2, 6))
        n = [int(v) for v in rng.integers(1, 400, d)]
        caps = [int(v) for v in rng.integers(1, 257, d - 1)]
        grid = [int(rng.integers(0, v + 1)) for v in n] if rng.random() < 0.7 else None
        for ranks in (caps, [1] * (d - 1), [int(rng.integers(1, c + 1)) for c in caps]):
            tiles, cap, bad = ttcross.check_tiles(n, ranks, caps, grid=grid, tile_edge=32, stored=True)
            assert bad == 0 and np.all(tiles <= cap), (n, ranks, caps, grid)
