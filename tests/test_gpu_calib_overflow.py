"""A calibration loss beyond FP32 is infinite, not NaN, and the gradients stay."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_calib import mw, problem, problem_jones  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [1, 5, 64, 200])  # one channel a warp, and several
def test_overflowing_loss(mw, C):  # noqa: F811
    """Residuals near 1e21: their squares, 1e42, are beyond FP32 (3.4e38), their
    products with the model are not.  (Gradient tolerance: that of the other
    calibration tests, 1e-4 of the largest.)"""
    V, M, g = problem(64, C, seed=C)
    V *= np.float32(1e20)
    Vd, Md, gd = (torch.from_numpy(a).cuda() for a in (V, M, g))
    loss, grad = mw.calib_loss_grad(Vd, Md, gd)
    want = oracle.calib_grad(V.astype(np.complex128), M.astype(np.complex128), g.astype(np.complex128))
    assert torch.isposinf(loss).item()
    assert np.abs(grad.cpu().numpy() - want).max() <= 1e-4 * np.abs(want).max()
    loss, grad = mw.calib_chan_loss_grad(Vd, Md, gd.repeat(C, 1))
    assert torch.isposinf(loss).item()
    assert np.abs(grad.cpu().numpy().sum(0) - want).max() <= 1e-4 * np.abs(want).max()
    V, M, J, _ = problem_jones(32, C, seed=C)
    V *= np.float32(1e20)
    loss, grad = mw.calib_jones_loss_grad(*(torch.from_numpy(a).cuda() for a in (V, M, J)))
    want = oracle.calib_jones_grad(V.astype(np.complex128), M.astype(np.complex128), J.astype(np.complex128))
    assert torch.isposinf(loss).item()
    assert np.abs(grad.cpu().numpy() - want).max() <= 1e-4 * np.abs(want).max()
