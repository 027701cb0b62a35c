"""Bounded waits of the fused mode's other kernels: 8-bit samples, the FP16 kind and
rows of 4-byte words.  The withheld release of test_gpu_failure.py, whose 4-bit whole
rows have a kernel of their own."""
import time

import pytest
import torch

import synth
from gpu_util import assert_exact, device_volt, oracle_for
from test_gpu_correlate import mw  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,N,fp16", [(8, 256, False), (8, 256, True), (8, 252, False), (8, 255, False), (4, 252, False)])
def test_withheld_release_times_out(mw, bits, N, fp16):  # noqa: F811
    spec = synth.Spec("fft", N, 400, 500, bits, seed=N, sigma=2 if bits == 4 else 20)
    kind = mw.KIND_FP16 if fp16 else mw.KIND_EXACT
    v = device_volt(spec)
    p = mw.Plan(N, 400, 500, bits, kind=kind, timeout_ms=150, test_fault=1)
    assert p.info().mma_shape == 4 and p.info().work_items > 2 * 152
    t0 = time.time()
    p.correlate(v)
    assert p.status() == mw.STATUS_BY_NAME["MWAX_ERR_TIMEOUT"]
    assert time.time() - t0 < 30.0
    p.close()
    q = mw.Plan(N, 400, 500, bits, kind=kind)
    got = q.correlate(v)[[0, 199, 399]].cpu().numpy()
    assert q.status() == 0
    assert_exact(got.astype("int64") if fp16 else got, oracle_for(spec, [0, 199, 399]), "after timeout")
    q.close()
    torch.cuda.synchronize()
