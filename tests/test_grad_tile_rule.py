"""The built-in shape of the mixed gradient (no GPU needed): lanes per system for
even planet counts, and never more of them than pairs of observations."""
import ctypes

import pytest


@pytest.mark.parametrize("n_pl", range(1, 9))
@pytest.mark.parametrize("n_obs", [1, 2, 3, 5, 8, 23, 24, 47, 48, 100])
def test_lanes(n_pl, n_obs):
    from paper_0812_2976_gb300 import _lib, build
    build.build()
    lib, tile = _lib.load(), _lib.KcTile()
    assert lib.kc_get_tile(1, 1, 200000, n_pl, n_obs, ctypes.byref(tile)) == 0
    G, block = tile.threads_per_system, tile.block
    least = {0: 8 if n_obs >= 48 else 4, 2: 4 if n_obs >= 24 or n_pl > 2 else 2}.get(n_pl % 4, 1)
    assert G & (G - 1) == 0 and 1 <= G <= 32 and block % G == 0 and block in (128, 256)
    assert G < max(2, n_obs)
    if n_obs > least:
        assert G >= least
