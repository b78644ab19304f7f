"""FP64 Matern jitters that keep a proposal's increments (gated stages) against jitters that draw
them again on acceptance (stage by stage): the same bits, for particles that accepted an odd number
of proposals (the increments end in the other buffer and are copied back) and an even number (they
do not), without and with a drift."""
import numpy as np
import pytest
import torch

from paper_2402_06927_gb300 import api
from paper_2402_06927_gb300.filter import EnsembleFilter

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,N", [(128, 100), (256, 40), (1024, 40)])
@pytest.mark.parametrize("drift", [False, True])
def test_kept_proposals_equal_redrawn(n, N, drift):
    g = api.SchModel(L=40.0, n=n, alpha=1.0, mu=0.02, dt=0.025, amps=[0.05], M=16, sigma=0.2, tol=1e-13, max_iter=60,
                     dtype="f64", noise="matern", kappa=1.0, eta=0.2)
    u0 = torch.linspace(0, 2 * np.pi, n + 1, device="cuda", dtype=torch.float64)[:-1].sin().mul(0.2).contiguous()
    m0, _ = g.prior_sample(N, u0, 4, 0.1)
    y = g.synth_obs(u0, 20, 1)
    lam = 0.3 * torch.randn((N, 4, n), generator=torch.Generator().manual_seed(6), dtype=torch.float64).cuda()
    fs = [EnsembleFilter(g, N, 4, 0.5 * N, 0.9, 4, 11, eager_stages=e) for e in (2, 0)]
    seen = set()
    for c in range(3):
        for f in fs:
            f.set_state(m0)
            if drift:
                f.set_drift(lam)
            f.cycle(y, c)
        for name in ("m_start", "m_end", "u_end", "dW", "nll", "logG", "accepts"):
            assert torch.equal(getattr(fs[0], name), getattr(fs[1], name)), name
        seen |= set(fs[0].accepts.tolist())
    assert seen & {1, 3} and seen & {2, 4}
