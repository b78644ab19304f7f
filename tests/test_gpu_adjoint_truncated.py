"""The reverse step that runs out of iterations: the FP64 adjoint then solves the step again by its
plain iteration, on the reloaded states and noise.  Its gradients are those of the transposed fixed
point truncated at the same count, formed here with numpy from the oracle's truncated states:

    P^T psi_k = g - (dt/2) M H^{-1} B^T psi_{k-1},  psi_0 = 0,
    dJ/dm0 = N^T psi - (dt/2) M H^{-1} B^T psi,  dJ/d(dU) = -B^T psi,

P, N = M +- (mu dt/2 K + 1/2 A_dv), B v = A(mbar, v).  Both sides are FP64 with the same operations
but for the order in the solves: 1e-10, as the truncated forward steps.
"""
import numpy as np
import pytest
import torch

from oracle.nudge import advection_in_v, obs_grad_u
from workloads import get_config, random_drift, random_increments, random_obs, random_state
from tests.helpers import gpu_model, oracle_model, rel_err, tdev

pytestmark = pytest.mark.gpu


def _transpose(tri):
    a, b, c = tri                        # rows a_i x_{i-1} + b_i x_i + c_i x_{i+1}
    return np.roll(c, 1), b, np.roll(a, -1)


def _truncated_gradients(om, m0, dW, lam, y, sigma, limit):
    m, u = m0, om.u_from_m(m0)
    traj = [(m, u)]
    for s in range(len(dW)):
        m, u, _, ok = om.step(m, u, om.noise(dW[s], lam[s]))
        assert not ok
        traj.append((m, u))
    M, K, Xi = om.mass(), om.stiffness(), om.noise_matrix()
    mh = lambda x: om.apply(M, om.solve(om.helmholtz(), x))   # noqa: E731  M H^{-1}
    g = mh(obs_grad_u(u, y, sigma))
    g_dW = np.empty_like(dW)
    for s in reversed(range(len(dW))):
        (ma, ua), (mb, ub) = traj[s], traj[s + 1]
        A = om.advection(0.5 * om.dt * (ua + ub) + om.noise(dW[s], lam[s]))
        half = [0.5 * om.mu * om.dt * k + 0.5 * a for k, a in zip(K, A)]
        P = _transpose([x + h for x, h in zip(M, half)])
        N = _transpose([x - h for x, h in zip(M, half)])
        B = advection_in_v(om, 0.5 * (ma + mb))
        corr = np.zeros_like(g)
        for _ in range(limit):
            psi = om.solve(P, g - corr)
            corr = 0.5 * om.dt * mh(B.T @ psi)
        g = om.apply(N, psi) - corr
        g_dW[s] = Xi.T @ -(B.T @ psi)
    return g_dW, om.dt * (g_dW + lam), g


@pytest.mark.parametrize("name,n", [("cfg1_f64", 128), ("cfg1_f64", 1024), ("cfg1m_f64", 128)])
@pytest.mark.parametrize("limit", [1, 2])
@pytest.mark.parametrize("ckpt", [None, 2])
def test_truncated_gradients(name, n, limit, ckpt):
    cfg = get_config(name, n=n, max_iter=limit)
    g, om = gpu_model(cfg), oracle_model(cfg)
    om.max_iter, om.tol = limit, cfg.tol
    m0 = np.stack([om.m_from_u(u) for u in random_state(cfg, 2, 3)])
    dW, lam = random_increments(cfg, 2, 4, steps=5), random_drift(cfg, 2, 7, steps=5)
    y = random_obs(cfg, 8, noise=0.05)
    out = g.adjoint_window(tdev(m0, g.dtype), tdev(dW, g.dtype), tdev(lam, g.dtype), tdev(y, g.dtype), ckpt=ckpt)
    torch.cuda.synchronize()
    assert torch.all(out["status"] == 1) and torch.all(out["iters"] == 2 * 5 * limit)
    for p in range(2):
        ref = _truncated_gradients(om, m0[p], dW[p], lam[p], y, cfg.sigma, limit)
        for k, r in zip(("g_dW", "g_lam", "g_m0"), ref):
            assert rel_err(out[k][p].cpu().numpy(), r) < 1e-10, k
