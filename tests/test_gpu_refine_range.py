"""FP64 steps by defect correction where the float side of an iteration ends: states so large
that the Helmholtz solve's right-hand side leaves the float range while m and its change stay
inside it (the time step is next to zero, so that the transport is the noise's alone and the step
is linear).  Such a step is run again by the plain FP64 iteration: m and u are the oracle's.
"""
import numpy as np
import pytest
import torch

from workloads import get_config, random_increments, random_state
from tests.helpers import gpu_model, oracle_model, rel_err, tdev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [128, 256, 1024])
def test_helmholtz_side_out_of_float_range(n):
    cfg = get_config("cfg1_f64", n=n, dt=1e-60)
    g, om = gpu_model(cfg), oracle_model(cfg)
    m0 = np.stack([om.m_from_u(u) for u in random_state(cfg, 2, 3)])
    m0 *= 1.2e38 / np.max(np.abs(m0))
    dW = random_increments(cfg, 2, 4, steps=1)
    dW *= 30.0 / np.max(np.abs(dW))
    ref = [om.step(m0[p], om.u_from_m(m0[p]), om.noise(dW[p, 0])) for p in range(2)]
    dm = max(np.max(np.abs(r[0] - m)) for r, m in zip(ref, m0))
    assert 6 * dm > 5e38 and dm < 2e38 and max(np.max(np.abs(r[0])) for r in ref) < 3e38
    out = g.ensemble_step(tdev(m0, g.dtype), tdev(dW, g.dtype))
    torch.cuda.synchronize()
    assert torch.all(out["status"] == 0)
    for p in range(2):
        assert rel_err(out["m"][p].cpu().numpy(), ref[p][0]) < 1e-11
        assert rel_err(out["u"][p].cpu().numpy(), ref[p][1]) < 1e-11
