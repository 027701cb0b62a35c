"""Tiles whose baselines leave the range of an int, or are not finite, reach no
cell of the grid, whichever coordinate it is."""
import numpy as np
import pytest

import oracle
from test_gpu_grid import close, gpu_grid, mw, problem  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W", [1, 6, 15])
@pytest.mark.parametrize("far", [4.3e9, -4.3e9, 8.6e9, 1e30, 1e300, np.inf, -np.inf, np.nan])
def test_far_tile(mw, far, W):  # noqa: F811
    """Metres are about half a cell here: 4.3e9 is a little over 2^31 cells, 8.6e9
    over 2^32.  The other baselines' sums are those of the array with that tile
    at a distance that an int holds, bit for bit, and the oracle's without it."""
    tile_xy, vis, f0, df = problem(W, 5, 4, 64, 1.0)
    k = 2
    ref_xy = tile_xy.copy()
    ref_xy[k] = [1e6, 1e6]
    ref, n_ref = gpu_grid(mw, ref_xy, vis, f0, df, 64, 1.0, W, 1.0)
    i = np.arange(10)
    own = np.isin(i // 2, [k])
    r, c = np.tril_indices(10)
    without = vis.copy()
    without[:, own[r] | own[c]] = 0
    close(ref, oracle.grid(tile_xy, without, f0, df, 64, 1.0, W, 1.0))
    for axis in ([0], [1], [0, 1]):
        xy = tile_xy.copy()
        xy[k, axis] = far
        got, n = gpu_grid(mw, xy, vis, f0, df, 64, 1.0, W, 1.0)
        assert n == n_ref and np.array_equal(got, ref)
