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


# ---- 8-bit samples in the fused pair mode (automatic above 64 MB of operands) ----------
@pytest.mark.parametrize("N,T,C,fp16", [
    (256, 2049, 35, False), (250, 2080, 33, False), (128, 1500, 94, True), (96, 4001, 35, True),
    (300, 2000, 24, False), (384, 513, 90, True), (131, 2111, 33, False), (640, 1000, 27, False),
    (255, 512, 140, False), (1000, 1400, 13, False)])
def test_fused_8bit(mw, N, T, C, fp16):  # noqa: F811
    """One to eight tiles, whole-unit and ragged rows (even and odd N), stage and
    block edges, one exact segment (T = 512) and checked ones; the FP16 kind is
    exact here too (every sum below 2^24)."""
    spec = synth.Spec("f8", N, C, T, 8, seed=N + 3 * T + C, sigma=20, tone_amp=3.0)
    p = mw.Plan(N, C, T, 8, kind=mw.KIND_FP16 if fp16 else mw.KIND_EXACT)
    inf = p.info()
    assert inf.mma_shape == 4 and inf.checked_segment == (0 if fp16 or T <= 512 else 1)
    v = device_volt(spec)
    out = p.correlate(v)
    out = p.correlate(v, out)
    assert p.status() == 0 and p.recomputed_channels() == 0
    chans = [0, 1, C // 2, C - 1]
    got = out.cpu().numpy()[chans]
    assert_exact(got.astype("int64") if fp16 else got, oracle_for(spec, chans), f"fused8 {N},{T},{C},{fp16}")
    p.close()


@pytest.mark.parametrize("N,group", [(256, 0), (250, 31), (129, 37)])
def test_fused_8bit_recompute(mw, N, group):  # noqa: F811
    """Full-scale channels leave the one-segment window: the check flags them,
    their operands are made from the rows and the narrow launch recomputes them;
    with all channels flagged the next calls unpack and run narrow."""
    import numpy as np
    import oracle
    import torch

    T, C = 2200, 40
    C = C if N > 200 else 74
    rng = np.random.default_rng(N)
    x = np.clip(np.rint(rng.normal(0, 20, (C, T, N, 2))), -127, 127).astype(np.int8)
    loud = [1, 24, C - 1]
    for c in loud:
        x[c] = rng.choice([-127, 127], (T, N, 2)).astype(np.int8)
    p = mw.Plan(N, C, T, 8, **({"chan_group": group} if group else {}))
    assert p.info().mma_shape == 4
    chans = loud + [0, 2, 23, 25, C - 2]
    v = torch.from_numpy(x.view(np.uint8).ravel().copy()).cuda()
    out = p.correlate(v)
    assert p.status() == 0
    assert p.recomputed_channels() == len(loud)
    ref = oracle.correlate(x[chans].view(np.uint8).ravel().copy(), 8, N, len(chans), T)
    assert_exact(out.cpu().numpy()[chans], ref, f"recompute {N}")
    x[:] = rng.choice([-127, 127], x.shape).astype(np.int8)
    v = torch.from_numpy(x.view(np.uint8).ravel().copy()).cuda()
    ref = oracle.correlate(x[chans].view(np.uint8).ravel().copy(), 8, N, len(chans), T)
    for want in (C, 0, 0):
        out = p.correlate(v)
        assert p.status() == 0
        assert p.recomputed_channels() == want
        assert_exact(out.cpu().numpy()[chans], ref, f"full scale {N}")
    p.close()
