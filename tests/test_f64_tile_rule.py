"""The built-in shape of the FP64 chi2 (no GPU needed): a warp per system or more
from 128 observations on, and at any size lanes and blocks the kernel takes."""
import ctypes

import pytest


@pytest.mark.parametrize("n_sys", [1, 300, 4096, 31298, 1 << 20])
@pytest.mark.parametrize("n_obs", [1, 2, 63, 127, 128, 639, 5000])
def test_lanes(n_sys, n_obs):
    from paper_0812_2976_gb300 import _lib, build
    build.build()
    lib, tile = _lib.load(), _lib.KcTile()
    for n_pl in (1, 4, 8):
        assert lib.kc_get_tile(0, 0, n_sys, n_pl, n_obs, ctypes.byref(tile)) == 0
        G, block = tile.threads_per_system, tile.block
        assert G & (G - 1) == 0 and block in (64, 128, 256) and block % G == 0 and tile.split == 0
        assert (32 if n_obs >= 128 else 1) <= G <= max(1, 2 * n_obs)
