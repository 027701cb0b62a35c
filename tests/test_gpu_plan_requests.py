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
