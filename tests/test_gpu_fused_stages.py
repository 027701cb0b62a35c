"""Pair-mode stages of three blocks (items of two tiles) and the automatic
choice of the fused pair mode beyond two tiles, bit-exact against the oracle.

T is chosen around whole blocks (64 samples at 4 bits, 32 at 8) so that an
item's last stage holds one, two or three blocks, and around whole stages."""
import pytest

import synth
from gpu_util import assert_exact, device_volt, oracle_for
from test_gpu_correlate import mw  # noqa: F401

pytestmark = pytest.mark.gpu


def check(mw, N, T, C, bits, what, **kw):  # noqa: F811
    spec = synth.Spec("st", N, C, T, bits, seed=N + 5 * T + C, sigma=2 if bits == 4 else 20, tone_amp=0.3)
    p = mw.Plan(N, C, T, bits, **kw)
    inf = p.info()
    out = p.correlate(device_volt(spec))
    assert p.status() == 0
    assert_exact(out.cpu().numpy(), oracle_for(spec, range(C)), f"{what} {N},{T},{C},{bits}")
    p.close()
    return inf


@pytest.mark.parametrize("blocks", [1, 2, 3, 4, 5, 6, 7, 13])
@pytest.mark.parametrize("N,C", [(96, 3), (128, 1), (256, 3), (384, 2)])
def test_fused_stage_edges(mw, blocks, N, C):  # noqa: F811
    """One, two and three tiles per item (a single diagonal item at C = 1)."""
    for T in (64 * blocks, 64 * blocks - 63):
        assert check(mw, N, T, C, 4, "fused", mma_shape=4).mma_shape == 4


@pytest.mark.parametrize("blocks", [1, 3, 4, 5, 6, 7])
@pytest.mark.parametrize("bits,N,C", [(8, 250, 3), (8, 256, 2), (4, 250, 3), (8, 100, 3), (8, 300, 2)])
def test_pair_stage_edges(mw, blocks, bits, N, C):  # noqa: F811
    """The pair mode's two-tile jobs (three-block stages) and a three-tile one."""
    S = 64 if bits == 4 else 32
    for T in (S * blocks, S * blocks - S + 1):
        assert check(mw, N, T, C, bits, "pair", mma_shape=3).mma_shape == 3


def test_fused_choice_beyond_two_tiles(mw):  # noqa: F811
    """Automatic: fused once the operands exceed 64 MB and an item has four
    blocks per tile; the pair mode just below either."""
    tile = 128 * 128  # operand bytes of a tile and block
    C = (64 << 20) // (3 * 12 * tile)  # three tiles, 12 blocks: 64 MB and a bit less
    assert check(mw, 384, 12 * 64, C + 1, 4, "auto").mma_shape == 4
    p = mw.Plan(384, C, 12 * 64, 4)
    assert p.info().mma_shape == 3
    p.close()
    p = mw.Plan(384, 2 * C, 11 * 64, 4)
    assert p.info().mma_shape == 3
    p.close()


@pytest.mark.parametrize("N,T,C,G", [
    (250, 2000, 140, 0), (129, 333, 700, 300), (115, 4097, 66, 0), (255, 1000, 66, 64), (17, 3000, 400, 0),
    (300, 1001, 200, 95), (497, 1100, 70, 0)])
def test_fused_ragged_rows(mw, N, T, C, G):  # noqa: F811
    """Sample rows that are not whole 16-byte units, copied to padded ones:
    every byte shift, channel groups that start inside a unit, odd N and T."""
    kw = {"chan_group": G} if G else {}
    spec = synth.Spec("rg", N, C, T, 4, seed=N + 5 * T + C, sigma=2, tone_amp=0.3)
    p = mw.Plan(N, C, T, 4, **kw)
    assert p.info().mma_shape == 4
    out = p.correlate(device_volt(spec))
    assert p.status() == 0
    chans = sorted({0, 1, C // 2, C - 2, C - 1} | ({G - 1, G} if G else set()))
    assert_exact(out.cpu().numpy()[chans], oracle_for(spec, chans), f"ragged {N},{T},{C},{G}")
    p.close()


def test_fused_batch_with_ragged_jobs(mw):  # noqa: F811
    """One persistent launch over whole-unit and ragged jobs; the graphs are
    built again for other buffers."""
    jobs = [(300, 40, 1500), (48, 5, 300), (256, 60, 3000), (33, 7, 999)]
    specs = [synth.Spec(f"rb{k}", n, c, t, 4, seed=70 + k, sigma=2, tone_amp=0.3) for k, (n, c, t) in enumerate(jobs)]
    bp = mw.BatchPlan(jobs, sample_bits=4)
    assert bp.info().mma_shape == 4
    for _ in range(2):
        vs = [device_volt(s) for s in specs]
        outs = bp.correlate(vs)
        assert bp.status() == 0
        for s, o in zip(specs, outs):
            chans = [0, s.n_chan // 2, s.n_chan - 1]
            assert_exact(o.cpu().numpy()[chans], oracle_for(s, chans), f"ragged batch {s.name}")
    bp.close()
