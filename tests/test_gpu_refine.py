"""FP64 steps by defect correction (float correction solves, double residuals): the
branches the other FP64 parity tests do not reach.

* A step that runs out of iterations is run again by the plain FP64 iteration, so a window
  with a small iteration limit must give the oracle's truncated iterates.
* The adjoint's float side is scaled by a power of two, so a gradient far outside the float
  range must come out as the exactly scaled gradient: J's misfit gradient scales with
  sigma^-2, and sigma a power of two scales every double operation exactly.
"""
import numpy as np
import pytest
import torch

from workloads import get_config, random_drift, random_increments, random_obs, random_state
from tests.helpers import gpu_model, oracle_model, rel_err, tdev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [128, 256, 1024, 2048])
@pytest.mark.parametrize("limit", [1, 2])
def test_truncated_step_is_the_plain_iteration(n, limit):
    cfg = get_config("cfg1_f64", n=n, max_iter=limit)
    g = gpu_model(cfg)
    om = oracle_model(cfg)
    om.max_iter, om.tol = limit, cfg.tol
    m0 = np.stack([om.m_from_u(u) for u in random_state(cfg, 2, 3)])
    dW = random_increments(cfg, 2, 4, steps=2)
    out = g.ensemble_step(tdev(m0, g.dtype), tdev(dW, g.dtype))
    torch.cuda.synchronize()
    assert np.all(out["status"].cpu().numpy() == 1)
    assert np.all(out["iters"].cpu().numpy() == 2 * limit)
    for p in range(2):
        m, u = m0[p], om.u_from_m(m0[p])
        for s in range(2):
            m, u, _, ok = om.step(m, u, om.noise(dW[p, s]))
            assert not ok
        assert rel_err(out["m"][p].cpu().numpy(), m) < 1e-10
        assert rel_err(out["u"][p].cpu().numpy(), u) < 1e-10


def _gradient(n, sigma_pow, **over):
    cfg = get_config("cfg1_f64", n=n, sigma=2.0 ** sigma_pow, **over)
    g = gpu_model(cfg)
    om = oracle_model(cfg)
    m0 = np.stack([om.m_from_u(u) for u in random_state(cfg, 2, 5)])
    y = random_obs(cfg, 8, noise=0.05)
    out = g.adjoint_window(tdev(m0, g.dtype), tdev(random_increments(cfg, 2, 6), g.dtype),
                           tdev(random_drift(cfg, 2, 7), g.dtype), tdev(y, g.dtype))
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("n", [128, 1024])
@pytest.mark.parametrize("power", [200, -200])
def test_gradient_scales_exactly(n, power):
    a, b = _gradient(n, 0), _gradient(n, power)
    assert torch.all(a["status"] == 0) and torch.equal(a["iters"], b["iters"])
    for k in ("g_dW", "g_m0"):
        assert torch.equal(a[k], b[k] * 2.0 ** (2 * power))


def test_truncated_adjoint_reports_it():
    out = _gradient(256, 0, max_iter=2)
    assert torch.all(out["status"] == 1)
    assert torch.all(out["iters"] == 4 * get_config("cfg1_f64").Ns)
    assert torch.all(torch.isfinite(out["g_dW"]))
