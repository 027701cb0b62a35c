"""Sizes of the gridding call's units and its two launches, which overlap where
few units are heavy.  Tolerance as in the strip walk's tests: 1e-5 of the largest
cell, ten times an FP32 sum's error at under 10^4 terms."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_grid import close, gpu_grid, mw, problem  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_tiles,n_chan,Ng,W", [
    (31, 22, 504, 5),    # 8 rows: under three units of 16 a warp
    (40, 120, 120, 7),   # 8 rows: under half a unit a warp, however dense
    (40, 140, 400, 6),   # over 40 entries a unit, few units: 16 rows
    (75, 90, 600, 5),    # over 40 entries a unit: 32
    (30, 60, 1068, 7),   # under four units (34 x 268) a warp: 16
    (20, 20, 1112, 7),   # four (35 x 279) of few entries: 32
    (50, 99, 1112, 7),   # over 8 entries: 16
    (20, 20, 1120, 13),  # two bands
])
def test_units(mw, n_tiles, n_chan, Ng, W):  # noqa: F811
    tile_xy, vis, f0, df = problem(Ng + W, n_tiles, n_chan, Ng, 1.0, spill=1.1)
    got, _ = gpu_grid(mw, tile_xy, vis, f0, df, Ng, 1.0, W, 0.16 * W)
    close(got, oracle.grid(tile_xy, vis, f0, df, Ng, 1.0, W, 0.16 * W))


@pytest.mark.parametrize("n_tiles,n_chan,Ng,W", [(20, 9, 256, 6), (24, 150, 64, 7)])
def test_calls_and_graphs_follow_one_another(mw, n_tiles, n_chan, Ng, W):  # noqa: F811
    """Other visibilities in every call, each call launched beside the last one's
    end, directly and from a captured graph: equal bit for bit to calls that wait."""
    tile_xy, vis, f0, df = problem(Ng, n_tiles, n_chan, Ng, 1.0)
    many = [torch.from_numpy(np.roll(vis, k, axis=1).copy()).cuda() for k in range(6)]
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        plan = mw.GridPlan(tile_xy, n_chan, f0, df, Ng, 1.0, W, 1.0)
        alone = []
        for v in many:
            alone.append(plan.grid(v).clone())
            s.synchronize()
        outs = [plan.empty_grids() for _ in many]
        for v, o in zip(many, outs):
            plan.grid(v, o)
        s.synchronize()
        assert all(torch.equal(a, o) for a, o in zip(alone, outs))
        v, o = many[0].clone(), plan.empty_grids()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            plan.grid(v, o)
        for k in (3, 1, 5):
            v.copy_(many[k])
            g.replay()
            g.replay()
            s.synchronize()
            assert torch.equal(o, alone[k])
        plan.close()
