"""Branches taken by size or by caller, each against the general form:

* tempering: the float location of the root and its FP64 Newton finish, at dead particles
  (infinite phi), two-valued phi, roots many octaves below the remaining step, and
  particle counts at the edges of a thread's share;
* resampling: weights at the ends of the quantisation (one, zero, subnormal, below 2^-50) and
  counts at the edges of a thread's share: the oracle's indices;
* FP64 windows and jitters of small launches (two-node chunks) against the same particles in a
  launch large enough for four-node chunks: both iterate to 1e-13, so a window of a few
  steps agrees to 1e-11 and the Metropolis decisions are the same;
* Matern jitters in gated stages (in FP64 they keep a proposal's increments) against stage by
  stage (drawn again on acceptance): the same bits.
"""
import numpy as np
import pytest
import torch

from oracle import filter as OF
from paper_2402_06927_gb300 import api
from paper_2402_06927_gb300.filter import EnsembleFilter
from workloads import get_config, random_obs, random_state
from tests.helpers import oracle_model, rel_err, tdev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [9, 33, 1024, 1025, 2049, 16384])
@pytest.mark.parametrize("kind", ["dead", "two", "far", "offset"])
@pytest.mark.parametrize("frac", [0.5, 0.9])
def test_temper_root_matches_oracle(N, kind, frac):
    rng = np.random.default_rng(N)
    phi = rng.gamma(2.0, 5.0, N)
    if kind == "dead":
        phi[1::7] = np.inf
        frac *= 0.8            # of all particles: six sevenths are alive
    elif kind == "two":
        phi = np.where(np.arange(N) % 3 == 0, 900.0, 1.0)
    elif kind == "far":
        phi = phi * 1e7
    else:
        phi = phi + 1e5
    w, out = api.pf_temper(tdev(phi, torch.float64), None, 0.25, frac * N)
    torch.cuda.synchronize()
    d, wb, e = OF.temper(phi, 0.25, frac * N, iters=90)
    assert abs(out[0].item() - d) <= 1e-12 * d * max(1.0, np.min(phi))   # d phi is rounded to its own size
    assert abs(out[1].item() - e) <= 1e-9 * e
    assert out[1].item() >= frac * N * (1 - 1e-12) or out[0].item() == 0.75 * 2.0 ** -60
    assert np.max(np.abs(w.cpu().numpy() - wb)) <= 1e-9 * np.max(wb)


@pytest.mark.parametrize("N", [1, 2, 1023, 1024, 1025, 2049, 8191, 8192])
@pytest.mark.parametrize("kind", ["one", "equal", "tiny", "spread"])
def test_resample_indices_match_oracle(N, kind):
    rng = np.random.default_rng(N)
    w = np.full(N, 1.0 / N)
    if kind == "one":
        w = np.zeros(N)
        w[N // 3] = 1.0
    elif kind == "tiny":
        w[::2] = rng.choice([0.0, 5e-324, 2.0 ** -51, 2.0 ** -50, 3.0 * 2.0 ** -51], w[::2].size)
        w[0] = 0.5
    elif kind == "spread":
        w = np.exp(-rng.gamma(2.0, 5.0, N))
    w = w / w.sum()
    for ctr in (0, 77):
        idx = api.pf_resample(tdev(w, torch.float64), 5, ctr)
        torch.cuda.synchronize()
        assert np.array_equal(idx.cpu().numpy(), OF.systematic_resample(w, OF.resample_offset(5, ctr)))


@pytest.mark.parametrize("noise", ["modes", "matern"])
@pytest.mark.parametrize("n", [128, 256])
def test_two_node_chunks_match_four(n, noise):
    cfg = get_config("cfg1_f64", n=n)
    kw = dict(noise=noise, kappa=1.0, eta=0.5) if noise == "matern" else {}
    g = api.SchModel(L=cfg.L, n=n, alpha=cfg.alpha, mu=cfg.mu, dt=cfg.dt,
                     amps=[0.05 / j for j in range(1, cfg.K // 2 + 1)], M=cfg.M, sigma=cfg.sigma, tol=1e-13,
                     max_iter=60, dtype="f64", **kw)
    om = oracle_model(cfg)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    N, big = 5, 3 * sms + 1
    m = tdev(np.stack([om.m_from_u(u) for u in random_state(cfg, N, 3)]), g.dtype)
    y = tdev(random_obs(cfg, 8), g.dtype)
    dW = g.draw_increments(N, 4, 3, 1, 0)
    rep = -(-big // N)
    outs = []
    for r in (1, rep):
        ms, ws = m.repeat(r, 1), dW.repeat(r, 1, 1)
        st = g.ensemble_step(ms, ws, None, y)
        acc, _, _ = g.jitter(ms, ws, None, y, st["nll"], st["logG"], st["m"], st["u"], 0.3, 0.9, 4, 5, 0)
        torch.cuda.synchronize()
        outs.append([v[:N].cpu().numpy() for v in (st["m"], st["u"], ws, st["nll"], acc, st["status"])])
    for a, b in zip(outs[0][:4], outs[1][:4]):
        assert rel_err(a, b) < 1e-11
    assert np.array_equal(outs[0][4], outs[1][4]) and np.array_equal(outs[0][5], outs[1][5])


@pytest.mark.parametrize("dtype,n,N", [("f32", 256, 40), ("f32", 1024, 24), ("f64", 128, 24), ("f64", 1024, 12)])
def test_matern_kept_proposals_equal_redrawn(dtype, n, N):
    g = api.SchModel(L=40.0, n=n, alpha=1.0, mu=0.02, dt=0.025, amps=[0.05], M=16, sigma=0.05,
                     tol=1e-6 if dtype == "f32" else 1e-13, max_iter=60, dtype=dtype, noise="matern", kappa=1.0,
                     eta=0.2)
    u0 = torch.linspace(0, 2 * np.pi, n + 1, device="cuda", dtype=torch.float64)[:-1].sin().mul(0.2).to(g.dtype)
    m0, _ = g.prior_sample(N, u0.contiguous(), 4, 0.1)
    y = g.synth_obs(u0.contiguous(), 20, 1)
    fs = [EnsembleFilter(g, N, 4, 0.5 * N, 0.9, 3, 11, eager_stages=e) for e in (2, 0)]
    for c in range(2):
        for f in fs:
            f.set_state(m0)
            f.cycle(y, c)
        for name in ("m_start", "m_end", "u_end", "dW", "nll", "logG", "accepts"):
            assert torch.equal(getattr(fs[0], name), getattr(fs[1], name)), name
