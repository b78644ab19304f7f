"""FP64 steps by defect correction over the Helmholtz length: alpha from a twentieth of a cell to
2000 cells (the float correction solve's condition grows with (alpha / h)^2).

u is corrected beside m and only m's change stops the iteration, so u is held to H^{-1} M m of the
returned m, formed by FFT (both matrices are circulant).  The bound: u's last correction belongs to
m's last change, at most 1e-13 max(1, max|m|), and the residual of H u = M m is rounded to a few
2^-53 of 6 (|m| + |u|), which H^{-1} scaled by (6 / h)^{-1} brings to the size of |m|: 4e-13 of
max|u| >= 0.5 max|m| >= 0.25 in all.  The gradient is held to a difference quotient.
"""
import numpy as np
import pytest
import torch

from workloads import get_config
from tests.helpers import gpu_model, tdev

pytestmark = pytest.mark.gpu


def _state(n, N):
    x = np.arange(n) * (40.0 / n)
    return np.stack([0.3 + 0.5 / np.cosh(x - 13.5 - 0.1 * p) + 0.1 * np.sin(2 * np.pi * 7 * x / 40.0) for p in range(N)])


@pytest.mark.parametrize("n", [128, 256, 512, 2048])
@pytest.mark.parametrize("ratio", [0.05, 1.0, 30.0, 300.0, 2000.0])
def test_velocity_is_that_of_the_momentum(n, ratio):
    cfg = get_config("cfg1_f64", n=n)
    g = gpu_model(cfg, alpha=ratio * cfg.h, max_iter=60)
    m = tdev(_state(n, 3), g.dtype)
    out = g.ensemble_step(m, g.draw_increments(3, 5, 3, 1, 0))
    torch.cuda.synchronize()
    assert torch.all(out["status"] == 0)
    th = 2 * np.pi * np.arange(n) / n
    mass, stiff = cfg.h * (2 + np.cos(th)) / 3, 4 * np.sin(th / 2) ** 2 / cfg.h
    me = out["m"].cpu().numpy()
    u = np.fft.ifft(np.fft.fft(me, axis=1) * (mass / (mass + (ratio * cfg.h) ** 2 * stiff)), axis=1).real
    assert np.max(np.abs(u)) >= 0.25
    assert np.max(np.abs(u - out["u"].cpu().numpy())) <= 4e-13 * np.max(np.abs(u))


@pytest.mark.parametrize("n", [128, 1024])
@pytest.mark.parametrize("ratio", [0.05, 30.0, 2000.0])
def test_gradient_is_the_difference_quotient(n, ratio):
    """dJ along a random direction of the increments: the central quotient at e = 1e-4 is off by e^2 J''' / 6
    (of the order of 1e-8 of J' here, where a direction moves u by its own size) and by the rounding
    of J over e, J 1e-13 / 1e-4 = 1e-9 J; 1e-5 of the gradient's scale bounds both."""
    cfg = get_config("cfg1_f64", n=n)
    g = gpu_model(cfg, alpha=ratio * cfg.h, max_iter=60)
    m = tdev(_state(n, 2), g.dtype)
    dW = g.draw_increments(2, 5, 3, 1, 0)
    y = torch.full((cfg.M,), 0.4, dtype=g.dtype, device="cuda")
    v = torch.randn(dW.shape, generator=torch.Generator().manual_seed(2), dtype=torch.float64).cuda()
    grad = g.adjoint_window(m, dW, torch.zeros_like(dW), y)["g_dW"]
    J = [g.ensemble_step(m, dW + e * v, None, y)["nll"] for e in (1e-4, -1e-4)]
    torch.cuda.synchronize()
    quotient, scale = (J[0] - J[1]) / 2e-4, (grad.abs() * v.abs()).sum((1, 2)) + (J[0] + J[1]).abs()
    assert torch.all(((grad * v).sum((1, 2)) - quotient).abs() <= 1e-5 * scale)
