"""What a plan is asked for and what it reports, where the automatic choice is
the fused pair mode."""
import pytest

import synth
from gpu_util import assert_exact, device_volt, oracle_for
from test_gpu_correlate import mw  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,N,T,C,G", [
    (8, 256, 2049, 70, 33), (8, 131, 2111, 66, 33), (4, 384, 768, 120, 115), (4, 250, 2000, 140, 70)])
def test_overlapped_pipeline_is_honoured(mw, bits, N, T, C, G):  # noqa: F811
    """pipeline 2 asks for an unpack that runs beside the correlation: the shape
    left to the plan is then one that unpacks."""
    spec = synth.Spec("ov", N, C, T, bits, seed=N + T, sigma=2 if bits == 4 else 20, tone_amp=0.3)
    p = mw.Plan(N, C, T, bits, chan_group=G)
    assert p.info().mma_shape == 4
    p.close()
    p = mw.Plan(N, C, T, bits, chan_group=G, pipeline=2)
    inf = p.info()
    assert inf.mma_shape == 3 and inf.pipeline == (1 if bits == 8 and N % 2 else 2)
    out = p.correlate(device_volt(spec))
    assert p.status() == 0
    chans = [0, G - 1, G, C - 1]
    assert_exact(out.cpu().numpy()[chans], oracle_for(spec, chans), f"overlapped {bits},{N}")
    p.close()


def test_overlapped_pipeline_keeps_small_arrays_fused(mw):  # noqa: F811
    """4-bit arrays of up to two tiles in whole rows have no unpack to overlap."""
    p = mw.Plan(256, 8, 2000, 4, chan_group=2, pipeline=2)
    assert p.info().mma_shape == 4 and p.info().pipeline == 1
    p.close()


@pytest.mark.parametrize("bits,N,C,blocks,shape", [
    (4, 640, 41, 20, 4), (4, 640, 40, 20, 3), (4, 640, 60, 19, 3),  # 5 tiles: 64 MB and 8 + 25 / 2 blocks
    (8, 896, 18, 32, 3), (8, 896, 18, 33, 4), (8, 896, 19, 32, 4),  # 7 tiles: 64 MB and 32 blocks
    (8, 896, 40, 31, 3),
    (4, 252, 65, 8, 4), (4, 252, 64, 8, 3),   # rows of words, two tiles: 16 MB
    (8, 372, 110, 13, 4), (8, 500, 200, 16, 3), (8, 501, 130, 16, 4),  # 8-bit rows of words: up to three tiles
])
def test_fused_lines(mw, bits, N, C, blocks, shape):  # noqa: F811
    """Both sides of each line of the automatic choice (a tile's block is 16 KB)."""
    p = mw.Plan(N, C, blocks * (64 if bits == 4 else 32), bits)
    assert p.info().mma_shape == shape
    p.close()


@pytest.mark.parametrize("N,T,C", [(256, 4000, 40), (250, 3000, 60), (255, 2500, 60)])
def test_fused_fp16_rounds_as_the_pair_mode(mw, N, T, C):  # noqa: F811
    """Full-scale samples, whose FP32 sums round: the same sums in the same order."""
    import torch

    gen = torch.Generator(device="cuda").manual_seed(N)
    v = (torch.randint(0, 2, (C * T * N * 2,), generator=gen, device="cuda") * 254 - 127).to(torch.int8).view(torch.uint8)
    p = mw.Plan(N, C, T, 8, kind=mw.KIND_FP16)
    q = mw.Plan(N, C, T, 8, kind=mw.KIND_FP16, mma_shape=3)
    assert p.info().mma_shape == 4 and q.info().mma_shape == 3
    a, b = p.correlate(v), q.correlate(v)
    assert p.status() == 0 and q.status() == 0
    assert a.max().item() > 2 ** 24 and torch.equal(a, b)
    p.close()
    q.close()
