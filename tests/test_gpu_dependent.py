"""Launches that start beside their predecessor: time ranges added into an output
that a kernel zeroes beside them, called again and again over a dirty output,
directly and from a captured graph (integer results: equal to the oracle's); a
solve's sweeps in one call and in several."""
import pytest
import torch

import synth
from gpu_util import assert_exact, device_volt, oracle_for
from test_gpu_correlate import mw  # noqa: F401

pytestmark = pytest.mark.gpu


def calls(mw, spec, **kw):  # noqa: F811
    p = mw.Plan(spec.n_inputs, spec.n_chan, spec.n_time, spec.sample_bits, **kw)
    volt = device_volt(spec)
    ref = oracle_for(spec, range(spec.n_chan))
    out = p.correlate(volt)
    assert p.status() == 0
    assert_exact(out.cpu().numpy(), ref, "first")
    for _ in range(3):
        out.fill_(-7)
        p.correlate(volt, out)
        p.correlate(volt, out)
    assert_exact(out.cpu().numpy(), ref, "again")
    g = torch.cuda.CUDAGraph()
    s = torch.cuda.Stream()
    q = mw.Plan(spec.n_inputs, spec.n_chan, spec.n_time, spec.sample_bits, stream=s, **kw)
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        q.correlate(volt, out)
        s.synchronize()
        with torch.cuda.graph(g, stream=s):
            q.correlate(volt, out)
        out.fill_(-7)
        g.replay()
        g.replay()
    torch.cuda.synchronize()
    assert p.status() == 0 and q.status() == 0
    assert_exact(out.cpu().numpy(), ref, "graph")
    q.close()
    p.close()


@pytest.mark.parametrize("bits,N,C,T", [
    (4, 64, 5, 700), (4, 100, 3, 900), (8, 48, 4, 300), (8, 250, 3, 290),
    (4, 512, 7, 257),
    (4, 512, 8, 257),  # more words than the zeroing kernel has threads
])
@pytest.mark.parametrize("shape", [0, 3])
def test_time_ranges(mw, bits, N, C, T, shape):  # noqa: F811
    spec = synth.Spec("dep", N, C, T, bits, seed=N + T, sigma=2 if bits == 4 else 20, tone_amp=0.3)
    calls(mw, spec, mma_shape=shape, k_split=2)


@pytest.mark.parametrize("gains", ["input", "chan", "jones"])
@pytest.mark.parametrize("N,C", [(4, 1), (64, 3), (100, 70), (256, 40)])
def test_sweeps_in_one_call_and_in_several(mw, gains, N, C):  # noqa: F811
    """Every pair of sweeps runs the same kernels: equal bit for bit."""
    gen = torch.Generator(device="cuda").manual_seed(N + C)
    size = {"input": (N,), "chan": (C, N), "jones": (N // 2, 2, 2)}[gains]
    solve = {"input": mw.calib_solve, "chan": mw.calib_chan_solve, "jones": mw.calib_jones_solve}[gains]
    cplx = lambda *s: torch.randn(*s, dtype=torch.complex64, device="cuda", generator=gen)  # noqa: E731
    V, M = cplx(C, N * (N + 1) // 2), cplx(C, N * (N + 1) // 2)
    g0 = cplx(*size) + (2 * torch.eye(2, device="cuda") if gains == "jones" else 2)
    whole, losses = solve(V, M, g0, 12)
    g, parts = g0, []
    for _ in range(6):
        g, h = solve(V, M, g, 2)
        torch.cuda.synchronize()
        parts.append(h)
    assert torch.isfinite(torch.view_as_real(whole)).all()
    assert torch.equal(whole, g) and torch.equal(losses, torch.cat(parts))
