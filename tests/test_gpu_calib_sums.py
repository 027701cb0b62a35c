"""The sums of the calibration passes at shapes with few channel groups."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_calib import mw, problem  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,C", [(1472, 100), (1024, 196), (768, 116)])
def test_jones_sums_take_no_longer_chains(mw, N, C):  # noqa: F811
    """Equal terms x of 17 bits: n of them add up exactly in FP32 while n is at
    most 128, and with a systematic error of about 5e-6 at 416.  A lane's
    uncompensated sum over the rows of a calibration tile and its warp's channels
    has 2 x 32 to 3 x 32 terms when twelve groups share the channels, so it is
    exact; what follows rounds at most 7 times (the warps' partials) and then
    adds compensated: 12 x 2^-24 of the sum of equal signs in all."""
    x = 127071 / 2 ** 17
    B = N * (N + 1) // 2
    M = torch.ones(C, B, dtype=torch.complex64, device="cuda")
    V = torch.full((C, B), 1 - x, dtype=torch.complex64, device="cuda")
    J = torch.eye(2, dtype=torch.complex64, device="cuda").repeat(N // 2, 1, 1)
    _, grad = mw.calib_jones_loss_grad(V, M, J)
    # G = sum over the other tiles and channels of R B^H (or R^H A) = 2 x in every entry
    want = 2 * 2 * x * (N // 2 - 1) * C
    err = (torch.view_as_real(grad).double() / want - torch.tensor([1.0, 0.0], device="cuda").double()).abs().max()
    assert err.item() <= 12 * 2.0 ** -24, err.item() * 2 ** 24


@pytest.mark.parametrize("N", [2, 32, 33, 479, 480, 481, 512, 513, 545])
def test_channel_gather_edges(mw, N):  # noqa: F811
    """One to eighteen blocks of 32 inputs: contributions around whole batches of sixteen.
    (1e-4 of the largest value, as in the other tests.)"""
    C = 3
    V, M, g = problem(N, C, seed=N)
    G = np.stack([g * np.exp(0.1j * c) for c in range(C)]).astype(np.complex64)
    Vd, Md, Gd = (torch.from_numpy(a).cuda() for a in (V, M, G))
    _, grad = mw.calib_chan_loss_grad(Vd, Md, Gd)
    new, _ = mw.calib_chan_solve(Vd, Md, Gd, 1)
    for c in range(C):
        v, m, g64 = (a.astype(np.complex128) for a in (V[c:c + 1], M[c:c + 1], G[c]))
        want = oracle.calib_grad(v, m, g64)
        assert np.abs(grad[c].cpu().numpy() - want).max() <= 1e-4 * np.abs(want).max()
        h, _ = oracle.calib_solve(v, m, g64, 1)
        assert np.abs(new[c].cpu().numpy() - h).max() <= 1e-4 * np.abs(h).max()


@pytest.mark.parametrize("N,C", [(512, 96), (510, 90)])
def test_jones_gather_loses_nothing(mw, N, C):  # noqa: F811
    """Whole residuals below 2^14 and a model of ones: every partial sum of the pass
    (at most 8 warps x 32 rows x 2 terms) is below 2^24 and exact, so what the gather
    rounds is all there is.  It carries what its additions lose: the nearest FP32
    number, where sixteen rounded sums miss it in every tenth entry."""
    gen = torch.Generator(device="cuda").manual_seed(N)
    n, B = N // 2, N * (N + 1) // 2
    R = torch.randint(1, 2 ** 14, (C, B), generator=gen, device="cuda")
    M = torch.ones(C, B, dtype=torch.complex64, device="cuda")
    J = torch.eye(2, dtype=torch.complex64, device="cuda").repeat(n, 1, 1)
    # M J^H = J M has 1 in every entry, and a model block of ones is J_a M J_b^H
    _, grad = mw.calib_jones_loss_grad((1 - R).to(torch.complex64), M, J)
    a, b = torch.tril_indices(n, n, -1, device="cuda")
    row = a * (2 * a + 1) + 2 * b
    r = R.sum(0).double()
    blk = torch.stack([r[row], r[row + 1], r[row + 2 * a + 1], r[row + 2 * a + 2]], 1).view(-1, 2, 2)
    G = torch.zeros(n, 2, dtype=torch.float64, device="cuda")
    G.index_add_(0, a, blk.sum(2))  # R B^H: row sums, the same in both columns
    G.index_add_(0, b, blk.sum(1))  # R^H A: column sums
    want = (2 * G).float()[:, :, None].expand(n, 2, 2)
    assert (grad.real == want).all().item() and (grad.imag == 0).all().item()
