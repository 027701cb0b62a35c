"""A plan can be asked for the shape that it reports."""
import pytest

import synth
from gpu_util import assert_exact, device_volt, oracle_for
from test_gpu_correlate import mw  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,N,T,C,fp16", [
    (8, 256, 2049, 35, False), (8, 250, 500, 140, False), (8, 255, 2080, 35, True), (4, 300, 1001, 70, False),
    (4, 115, 4097, 20, False), (4, 48, 100, 3, False), (4, 384, 300, 3, False), (8, 100, 700, 3, False)])
def test_reported_shape_can_be_asked_for(mw, bits, N, T, C, fp16):  # noqa: F811
    spec = synth.Spec("rs", N, C, T, bits, seed=N + T, sigma=2 if bits == 4 else 20, tone_amp=0.3)
    kind = mw.KIND_FP16 if fp16 else mw.KIND_EXACT
    p = mw.Plan(N, C, T, bits, kind=kind)
    inf = p.info()
    p.close()
    q = mw.Plan(N, C, T, bits, kind=kind, mma_shape=inf.mma_shape, chan_group=inf.chan_group, k_split=inf.k_split)
    asked = q.info()
    assert (asked.mma_shape, asked.checked_segment) == (inf.mma_shape, inf.checked_segment)
    out = q.correlate(device_volt(spec))
    assert q.status() == 0
    got = out.cpu().numpy()[[0, C - 1]]
    assert_exact(got.astype("int64") if fp16 else got, oracle_for(spec, [0, C - 1]), f"asked {bits},{N}")
    q.close()
    # and with its work items in two time ranges, as a tuner may ask (at most half the time blocks)
    if inf.mma_shape == 4 and not fp16 and T >= 4 * (64 if bits == 4 else 32):
        q = mw.Plan(N, C, T, bits, mma_shape=4, k_split=2)
        assert q.info().mma_shape == 4 and q.info().k_split == 2
        got = q.correlate(device_volt(spec)).cpu().numpy()[[0, C - 1]]
        assert q.status() == 0
        assert_exact(got, oracle_for(spec, [0, C - 1]), f"two ranges {bits},{N}")
        q.close()


def test_batch_shape_can_be_asked_for(mw):  # noqa: F811
    jobs = [(300, 40, 1500), (48, 5, 300), (256, 60, 3000), (33, 7, 999)]
    p = mw.BatchPlan(jobs, sample_bits=4)
    shape = p.info().mma_shape
    p.close()
    q = mw.BatchPlan(jobs, sample_bits=4, mma_shape=shape)
    assert shape == 4 and q.info().mma_shape == 4
    q.close()
