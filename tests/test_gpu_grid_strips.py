"""The strip walk of the gridding call against the FP64 oracle where it can go
wrong: one band and several (W = 1 .. 31), windows of five and seven rows,
grids whose half plane is not a whole number of strips, columns that are not
whole blocks, strips dense enough to be cut up and shared by a CTA, sparse
ones that are joined, points
past every edge and points exactly on the mirror row and column.

Tolerance: an FP32 sum of n terms in a fixed order is off by at most about
n 2^-24 of the sum of their magnitudes, in the mean sqrt(n) 2^-24; the densest
cells here sum under 10^4 terms of comparable size, so 1e-5 of the largest
cell leaves a factor of ten."""
import numpy as np
import pytest

import oracle
from test_gpu_grid import close, gpu_grid, mw, problem  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_tiles,n_chan,Ng,W,sigma,spill", [
    (3, 2, 8, 1, 0.5, 0.7),       # smallest grid and support
    (6, 5, 18, 2, 0.6, 1.4),      # even support, Ng not a multiple of 4
    (6, 5, 30, 3, 0.7, 1.4),
    (9, 7, 66, 4, 1.0, 1.2),      # 34 half-plane rows: a strip of two rows at the end
    (9, 7, 62, 5, 1.0, 1.2),      # 32 half-plane rows
    (9, 7, 64, 6, 1.0, 1.6),
    (9, 7, 100, 8, 1.2, 1.3),     # two bands
    (7, 6, 54, 14, 3.0, 1.5),     # two full bands
    (7, 6, 90, 15, 3.0, 1.2),     # three bands
    (5, 4, 80, 31, 6.0, 1.4),     # five bands, the largest support
    (24, 40, 16, 7, 1.0, 0.9),    # dense: every strip cut up, CTA-wide ones
    (24, 60, 40, 5, 0.8, 0.6),
    (5, 3, 262, 7, 1.0, 1.2),     # sparse: joined strips of 32 columns, a short last one
    (5, 3, 512, 9, 1.2, 1.2),     # the same in two bands
    (16, 9, 256, 6, 0.8, 1.6),    # both kinds beside each other
])
def test_strips(mw, n_tiles, n_chan, Ng, W, sigma, spill):  # noqa: F811
    tile_xy, vis, f0, df = problem(Ng * 100 + W, n_tiles, n_chan, Ng, 1.0, spill=spill)
    got, n = gpu_grid(mw, tile_xy, vis, f0, df, Ng, 1.0, W, sigma)
    close(got, oracle.grid(tile_xy, vis, f0, df, Ng, 1.0, W, sigma))
    assert 0 < n <= n_tiles * (n_tiles - 1) * n_chan


@pytest.mark.parametrize("W", [6, 7])
def test_points_on_the_mirror_axes(mw, W):  # noqa: F811
    """Tiles on a cross: baselines with no east or no north component lie on
    the middle row and column, whose cells are their own mirror images."""
    _, vis, f0, df = problem(3, 6, 4, 64, 1.0)
    tile_xy = np.array([[0.0, 0.0], [11.0, 0.0], [-23.0, 0.0], [0.0, 17.0], [0.0, -29.0], [0.0, 0.0]])
    got, _ = gpu_grid(mw, tile_xy, vis, f0, df, 64, 1.0, W, 1.0)
    close(got, oracle.grid(tile_xy, vis, f0, df, 64, 1.0, W, 1.0))
