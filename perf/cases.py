"""The performance cases of this framework: what its users have it do, through its public entry points.

A user of the particle filter runs assimilation cycles (forecast, tempering, resampling, PCN jitter),
plain forecasts, gradients of the window cost, the nudging optimiser, the learned drift's network
(inference and training) and the weight and resampling calls by themselves.  ``listed`` has one case
for each of these at the sizes of this repository's workloads and benchmark modes, or near them at
ragged sizes; ``draw`` gives more of the same kinds over the same ranges.

Kinds (a case's "kind"):
  cycle     EnsembleFilter.cycle from a given start ensemble (FP64 and FP32, mode and Matern noise)
  forecast  SchModel.ensemble_step with a nudging drift and the fused likelihood
  gradient  SchModel.adjoint_window, or NudgingCost through autograd
  nudge     SchModel.nudge, open-loop schedule (what generates the network's training pairs)
  net       ProposalNet.forward
  train     ProposalNet.loss_and_grad and adam_step (the body of train_step)
  weights   pf_temper, pf_resample and pf_gather_rows on an ensemble's rows

The inputs and the 64-bit values of ``exact`` come from plain torch: circulant matrices are applied
and inverted by FFT, implicit steps are iterated to their fixed point, gradients use autograd.
"""
from __future__ import annotations

import math

import torch

from paper_2402_06927_gb300.api import (NudgingCost, ProposalNet, SchModel, pf_gather_rows, pf_resample, pf_temper)
from paper_2402_06927_gb300.filter import EnsembleFilter

LENGTH, ALPHA, MU, DT = 40.0, 1.0, 0.02, 0.025   # the workloads' domain, Helmholtz length, viscosity, step
KAPPA, MATERN_K = 1.0, 3                         # the Matern noise's inverse length and chained solves


def listed():
    return [
        # the plain method in FP64 (n = 256, N = 32, 5-step windows): the smallest filter a user runs;
        # a cycle is a chain of short launches
        dict(name="cycle_f64_small", kind="cycle", dtype="f64", noise="modes", n=256, K=4, M=32, N=32, Ns=5,
             n_jitter=5, rho=0.8605, sigma=0.05, eta=0.0),
        # Exp 1's filter: the paper's Matern noise, 150 particles, n = 128, FP64
        dict(name="cycle_f64_matern", kind="cycle", dtype="f64", noise="matern", n=128, K=4, M=64, N=150, Ns=5,
             n_jitter=5, rho=0.8605, sigma=0.05, eta=1.0),
        # the ensemble-scale filter in FP32: n = 1024, N = 1024, ten proposals a stage
        dict(name="cycle_f32", kind="cycle", dtype="f32", noise="modes", n=1024, K=8, M=64, N=1024, Ns=10,
             n_jitter=10, rho=0.9999, sigma=0.05, eta=0.0),
        # the same ensemble with the Matern noise (one Brownian motion per cell)
        dict(name="cycle_f32_matern", kind="cycle", dtype="f32", noise="matern", n=1024, K=8, M=64, N=1024, Ns=10,
             n_jitter=10, rho=0.9999, sigma=0.05, eta=0.2),
        # the large run: n = 4096, N = 8192, the default benchmark's cycle
        dict(name="cycle_f32_large", kind="cycle", dtype="f32", noise="modes", n=4096, K=32, M=128, N=8192, Ns=10,
             n_jitter=10, rho=0.9999, sigma=0.02, eta=0.0),
        # a forecast of an odd-sized ensemble under a nudging drift, with the likelihood and Girsanov weight
        dict(name="forecast_f32_ragged", kind="forecast", dtype="f32", noise="modes", n=512, K=16, M=32, N=777, Ns=7,
             sigma=0.05, eta=0.0, drift=True),
        # gradients of the window cost in FP64, every state of the window kept
        dict(name="gradient_f64", kind="gradient", dtype="f64", n=1024, K=8, M=64, N=256, Ns=20, ckpt=0,
             sigma=0.05, autograd=False),
        # the same in FP32 for an odd ensemble, through autograd, checkpoints every 7 steps
        dict(name="gradient_f32_ragged", kind="gradient", dtype="f32", n=1024, K=16, M=64, N=301, Ns=17, ckpt=7,
             sigma=0.05, autograd=True),
        # the nudging optimiser that generates the learned drift's training pairs
        dict(name="nudge_f32", kind="nudge", dtype="f32", n=1024, K=16, M=64, N=512, Ns=20, sigma=0.05,
             max_iter=30, gtol=1e-4),
        # the learned drift of a whole ensemble
        dict(name="net_bf16", kind="net", n=1024, K=16, Ns=20, M=64, C=64, B=8192, sigma=0.05, precision="bf16"),
        # one training step at the training batch
        dict(name="train_bf16", kind="train", n=1024, K=16, Ns=20, M=64, C=64, B=256, sigma=0.05, precision="bf16"),
        # tempering, resampling and the gathers of a large ensemble's rows
        dict(name="weights_ragged", kind="weights", dtype="f32", n=1024, K=16, N=8001, Ns=10, spread=5.0, ess=0.5),
    ]


def _between(rng, lo, hi):
    """A whole number, spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["cycle", "cycle", "forecast", "gradient", "nudge", "net", "train", "weights"])
    if kind == "cycle":
        which = rng.choice(["f64", "f64", "f32", "f32", "large"])
        noise = rng.choice(["modes", "matern"]) if which != "large" else "modes"
        if which == "f64":
            n = rng.choice([128, 256, 512])
            return dict(kind=kind, dtype="f64", noise=noise, n=n, K=2 * rng.randint(1, 6),
                        M=n // rng.choice([2, 4, 8]), N=_between(rng, 16, 76800 // n), Ns=rng.randint(3, 8),
                        n_jitter=rng.randint(3, 6), rho=rng.choice([0.8605, 0.95, 0.99]), sigma=0.05,
                        eta=rng.choice([0.2, 1.0]) if noise == "matern" else 0.0)
        if which == "f32":
            n = rng.choice([256, 512, 1024])
            return dict(kind=kind, dtype="f32", noise=noise, n=n, K=2 * rng.randint(2, 10), M=n // 16,
                        N=_between(rng, 64, 2048), Ns=rng.randint(5, 12), n_jitter=rng.randint(5, 10), rho=0.9999,
                        sigma=0.05, eta=0.2 if noise == "matern" else 0.0)
        n = rng.choice([2048, 4096])
        return dict(kind=kind, dtype="f32", noise="modes", n=n, K=2 * rng.randint(4, 18), M=128,
                    N=_between(rng, 128, 4096), Ns=rng.randint(5, 10), n_jitter=rng.randint(5, 10), rho=0.9999,
                    sigma=0.02, eta=0.0)
    if kind == "forecast":
        dtype = rng.choice(["f32", "f32", "f64"])
        noise = rng.choice(["modes", "modes", "matern"])
        n = rng.choice([256, 512, 1024, 2048, 4096]) if dtype == "f32" else rng.choice([128, 256, 512, 1024])
        return dict(kind=kind, dtype=dtype, noise=noise, n=n, K=2 * rng.randint(1, 16), M=n // rng.choice([4, 8, 16]),
                    N=_between(rng, 16, 4096 if dtype == "f32" else 300), Ns=rng.randint(3, 12), sigma=0.05,
                    eta=0.2 if noise == "matern" else 0.0, drift=rng.random() < 0.5)
    if kind == "gradient":
        dtype = rng.choice(["f32", "f64"])
        n = rng.choice([256, 512, 1024, 2048])
        Ns = rng.randint(5, 20)
        return dict(kind=kind, dtype=dtype, n=n, K=2 * rng.randint(2, 10), M=n // 16,
                    N=_between(rng, 16, 1000 if dtype == "f32" else 262144 // n), Ns=Ns,
                    ckpt=rng.choice([0, 0, 3, 5]), sigma=0.05, autograd=rng.random() < 0.5)
    if kind == "nudge":
        n = rng.choice([256, 512, 1024])
        return dict(kind=kind, dtype="f32", n=n, K=2 * rng.randint(2, 8), M=n // 16, N=_between(rng, 32, 512),
                    Ns=rng.randint(5, 20), sigma=0.05, max_iter=30, gtol=1e-4)
    if kind in ("net", "train"):
        n = rng.choice([256, 1024, 1024, 2048])
        big = 1024 if n <= 1024 else 512
        return dict(kind=kind, n=n, K=2 * rng.randint(2, 10), Ns=rng.randint(5, 20), M=n // 16, C=64,
                    B=_between(rng, 16, 8 * big if kind == "net" else big), sigma=0.05,
                    precision=rng.choice(["bf16", "bf16", "bf16", "fp32"]))
    return dict(kind="weights", dtype="f32", n=rng.choice([256, 512, 1024, 4096]), K=2 * rng.randint(2, 16),
                N=_between(rng, 32, 8192), Ns=rng.randint(3, 12), spread=rng.choice([0.5, 5.0, 50.0]),
                ess=rng.choice([0.25, 0.5, 0.8]))


# ---------------------------------------------------------------------------------------------
# plain torch: the discretisation in 64 bits
# ---------------------------------------------------------------------------------------------
class _Mesh:
    """Periodic P1 matrices on n nodes, applied and inverted through their Fourier symbols."""

    def __init__(self, n):
        self.n, self.h = n, LENGTH / n
        th = 2 * math.pi * torch.arange(n // 2 + 1, dtype=torch.float64, device="cuda") / n
        self.mass = self.h / 6 * (4 + 2 * torch.cos(th))
        self.stiff = (2 - 2 * torch.cos(th)) / self.h
        self.helm = self.mass + ALPHA ** 2 * self.stiff
        self.pic = self.mass + 0.5 * MU * DT * self.stiff
        self.x = torch.arange(n, dtype=torch.float64, device="cuda") * self.h

    def apply(self, symbol, v):
        return torch.fft.irfft(symbol * torch.fft.rfft(v), n=self.n)

    def u(self, m):
        return self.apply(self.mass / self.helm, m)

    def m(self, u):
        return self.apply(self.helm / self.mass, u)

    def increment(self, case, w):
        """dU at the nodes from w = dW + lambda dt, [N, Q]."""
        if case.get("noise") == "matern":
            load = case["eta"] * math.sqrt(self.h) / 2 * (w.roll(1, -1) + w)
            g = self.mass + self.stiff / KAPPA ** 2
            return self.apply(self.mass ** (MATERN_K - 1) / g ** MATERN_K, load)
        j = torch.arange(1, case["K"] // 2 + 1, dtype=torch.float64, device="cuda")
        ang = 2 * math.pi / LENGTH * j[:, None] * self.x
        a = (0.05 / j)[:, None]
        modes = torch.stack([a * torch.sin(ang), a * torch.cos(ang)], 1).reshape(case["K"], self.n)
        return w @ modes

    def residual(self, m1, m0, dU):
        """R(m1; m0, dU) of the implicit midpoint step."""
        mb = 0.5 * (m0 + m1)
        dv = DT * self.u(mb) + dU
        right = mb + mb.roll(-1, -1)
        adv = 0.5 * (dv.roll(-1, -1) * right - dv.roll(1, -1) * right.roll(1, -1))
        return self.apply(self.mass, m1 - m0) + self.apply(MU * DT * self.stiff, mb) + adv

    def step(self, m0, dU, tol):
        m1 = m0
        for _ in range(300):
            d = self.apply(1 / self.pic, self.residual(m1, m0, dU))
            m1 = m1 - d
            if float(d.abs().max()) <= tol * max(1.0, float(m1.abs().max())):
                break
        return m1


def _profile(x):
    return 0.2 / torch.cosh(x - 27.0) + 0.5 / torch.cosh(x - 13.0)


def _ensemble(mesh, N, g):
    """Momenta of N smooth perturbations of the workloads' initial profile, [N, n] in 64 bits."""
    u = _profile(mesh.x) + 0.05 * torch.randn(N, 1, generator=g, dtype=torch.float64, device="cuda")
    for j in range(1, 5):
        a = 0.05 / j * torch.randn(2, N, 1, generator=g, dtype=torch.float64, device="cuda")
        ang = 2 * math.pi * j / LENGTH * mesh.x
        u = u + a[0] * torch.sin(ang) + a[1] * torch.cos(ang)
    return mesh.m(u)


def _noise_dim(case):
    return case["n"] if case.get("noise") == "matern" else case["K"]


def _increments(case, N, g):
    z = torch.randn(N, case["Ns"], _noise_dim(case), generator=g, dtype=torch.float64, device="cuda")
    return math.sqrt(DT) * z


def _observe(case, mesh, m, g):
    """Noisy observations of the window's end state of one truth, started at momentum m [1, n]."""
    w = _increments(case, 1, g)
    for s in range(case["Ns"]):
        m = mesh.step(m, mesh.increment(case, w[:, s]), 1e-11)
    z = torch.randn(case["M"], generator=g, dtype=torch.float64, device="cuda")
    return mesh.u(m)[0, :: case["n"] // case["M"]] + case["sigma"] * z


def _real(case):
    return torch.float32 if case["dtype"] == "f32" else torch.float64


def _inputs(case, seed):
    """Start momenta, increments, drift and observations of a window, in the case's precision."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    mesh = _Mesh(case["n"])
    m = _ensemble(mesh, case["N"] + 1, g)
    y = _observe(case, mesh, m[:1], g)
    dW = _increments(case, case["N"], g) if case["kind"] in ("forecast", "gradient") else None
    lam = None
    if case["kind"] == "gradient" or case.get("drift"):
        lam = 0.3 * torch.randn(dW.shape, generator=g, dtype=torch.float64, device="cuda")
    t = _real(case)
    return tuple(None if v is None else v.to(t).contiguous() for v in (m[1:], dW, lam, y))


def _net_inputs(case, seed):
    """The network's parameters and a batch: start velocities, observations, target drifts, Adam's moments."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    n, K, Ns, C, B = case["n"], case["K"], case["Ns"], case["C"], case["B"]
    mesh = _Mesh(n)
    u = mesh.u(_ensemble(mesh, B, g)).float().contiguous()
    rand = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    y = (_profile(mesh.x)[:: n // case["M"]].float() + case["sigma"] * rand(B, case["M"])).contiguous()
    if case["kind"] == "net":
        y = y[0].contiguous()      # one cycle's observations, shared by the ensemble
    parts, cin = [], 2
    for _ in range(4):
        parts += [rand(C * cin * 5) * (2.0 / (cin * 5)) ** 0.5, 0.05 * rand(C)]
        cin = C
    parts += [rand(K * Ns * C * K) * (1.0 / (C * K)) ** 0.5, 0.05 * rand(K * Ns)]
    params = torch.cat(parts)
    target = 0.3 * rand(B, Ns, K)
    moments = (1e-3 * rand(params.numel()), 1e-6 * (0.5 + rand(params.numel()).square()))
    return params, u, y, target, moments


def _model(case):
    f64 = case["dtype"] == "f64"
    n = case["n"]
    return SchModel(L=LENGTH, n=n, alpha=ALPHA, mu=MU, dt=DT, amps=[0.05 / j for j in range(1, case["K"] // 2 + 1)],
                    M=case.get("M", n // 16), sigma=case.get("sigma", 0.05), tol=1e-13 if f64 else 1e-6,
                    max_iter=60 if f64 else 100, dtype=case["dtype"], noise=case.get("noise", "modes"), kappa=KAPPA,
                    eta=case.get("eta", 1.0), matern_k=MATERN_K)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, seed=seed)
    if kind in ("net", "train"):
        params, u, y, target, (m, v) = _net_inputs(case, seed)
        net = ProposalNet(case["n"], case["K"], case["Ns"], case["M"], case["sigma"], C=case["C"], params=params,
                          precision=case["precision"])
        if kind == "train":        # in the middle of a training run
            net.m.copy_(m)
            net.v.copy_(v)
            net.t = 100
        st.update(net=net, u=u, y=y, target=target)
        return st
    if kind == "weights":
        g = torch.Generator(device="cuda").manual_seed(seed)
        N, n, dt = case["N"], case["n"], _real(case)
        e = torch.rand(2, N, generator=g, dtype=torch.float64, device="cuda")
        nll = -case["spread"] * (torch.log1p(-e[0]) + torch.log1p(-e[1]))
        logG = 0.3 * torch.randn(N, generator=g, dtype=torch.float64, device="cuda")
        rows = [torch.randn(s, generator=g, dtype=dt, device="cuda") for s in
                ((N, n), (N, n), (N, n), (N, case["Ns"], case["K"]))]
        st.update(nll=nll, logG=logG, src=rows, dst=[torch.empty_like(r) for r in rows])
        return st
    m, dW, lam, y = _inputs(case, seed)
    model = _model(case)
    st.update(model=model, m=m, dW=dW, lam=lam, y=y)
    if kind == "cycle":
        st["filter"] = EnsembleFilter(model, case["N"], case["Ns"], 0.5 * case["N"], case["rho"], case["n_jitter"],
                                      seed)
    return st


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "cycle":
        f = st["filter"]
        f.set_state(st["m"])
        f.cycle(st["y"], 0)
        return dict(m=f.m_end, u=f.u_end, dW=f.dW, nll=f.nll, logG=f.logG, accepts=f.accepts, status=f.status)
    if kind == "forecast":
        out = st["model"].ensemble_step(st["m"], st["dW"], st["lam"], st["y"], want_iters=False)
        return {k: out[k] for k in ("m", "u", "nll", "logG", "status")}
    if kind == "gradient":
        ckpt = case["ckpt"] or None
        if case["autograd"]:
            v = [st[k].detach().requires_grad_() for k in ("m", "dW", "lam")]
            J = NudgingCost.apply(st["model"], *v, st["y"], ckpt)
            J.sum().backward()
            return dict(J=J.detach(), g_m0=v[0].grad, g_dW=v[1].grad, g_lam=v[2].grad)
        out = st["model"].adjoint_window(st["m"], st["dW"], st["lam"], st["y"], ckpt=ckpt)
        return {k: out[k] for k in ("J", "g_m0", "g_dW", "g_lam")}
    if kind == "nudge":
        out = st["model"].nudge(st["m"], st["y"], case["Ns"], mode="open_loop", max_iter=case["max_iter"],
                                gtol=case["gtol"], seed=st["seed"])
        return {k: out[k] for k in ("lam", "dW", "J", "status")}
    if kind == "net":
        return st["net"].forward(st["u"], st["y"])
    if kind == "train":
        net = st["net"]
        loss, grads = net.loss_and_grad(st["u"], st["y"], st["target"])
        net.adam_step(grads, 1e-3)
        return dict(loss=loss, grads=grads, params=net.params, m=net.m, v=net.v)
    wbar, out = pf_temper(st["nll"], st["logG"], 0.0, case["ess"] * case["N"])
    idx = pf_resample(wbar, st["seed"], 0)
    return dict(wbar=wbar, out=out, idx=idx, rows=[pf_gather_rows(idx, s, d) for s, d in zip(st["src"], st["dst"])])


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------
def _net_flops(case):
    """2 flops per multiply-add of the forward contractions, one sample."""
    C, n, K, O = case["C"], case["n"], case["K"], case["K"] * case["Ns"]
    conv = sum((n >> (l + 1)) * C * 5 * (2 if l == 0 else C) for l in range(4))
    return 2.0 * (conv + C * (n // 16) * K + O * C * K)


def _net_params(case):
    C, K, O = case["C"], case["K"], case["K"] * case["Ns"]
    return 5 * C * (2 + 3 * C) + 4 * C + O * C * K + O


def work(case):
    kind = case["kind"]
    if kind in ("net", "train"):
        B, O, p = case["B"], case["K"] * case["Ns"], _net_params(case)
        if kind == "net":
            return dict(bytes=4.0 * (B * (case["n"] + O) + case["M"] + p), flops=B * _net_flops(case))
        # forward, input gradients and weight gradients; Adam reads g, p, m, v and writes p, m, v
        return dict(bytes=4.0 * (B * (case["n"] + O + case["M"]) + 8 * p), flops=3 * B * _net_flops(case) + 12.0 * p)
    w = 4 if case["dtype"] == "f32" else 8
    n, N, Ns, Q = case["n"], case["N"], case["Ns"], _noise_dim(case)
    if kind == "weights":
        return dict(bytes=2.0 * w * N * (3 * n + Ns * case["K"]) + 8.0 * 4 * N, flops=40.0 * N)
    # a step of one node: the noise, about four 30-flop iterations in FP32 and seven 44-flop ones in FP64
    step = (30 if case.get("noise") == "matern" else 2 * case["K"]) + (4 * 30 if w == 4 else 7 * 44)
    fields = 4.0 * w * N * n + w * N * Ns * Q
    if kind == "cycle":     # the forecast and one stage of proposals
        return dict(bytes=fields, flops=float(N) * Ns * n * step * (1 + case["n_jitter"]))
    if kind == "forecast":
        return dict(bytes=fields, flops=float(N) * Ns * n * step)
    back = 2 * case["K"] + 16 + (4 if w == 4 else 7) * 32
    if kind == "gradient":
        return dict(bytes=2.0 * w * N * n + 4.0 * w * N * Ns * Q, flops=float(N) * Ns * n * (step + back))
    return dict(bytes=w * N * (n + 2.0 * Ns * Q), flops=5.0 * N * Ns * n * (step + back))   # about four iterations


# ---------------------------------------------------------------------------------------------
# the values in 64 bits
# ---------------------------------------------------------------------------------------------
def _window(case, mesh, m, dW, lam, tol):
    """The states after each step, from momentum m."""
    w = dW if lam is None else dW + DT * lam
    ms = [m]
    dUs = []
    for s in range(case["Ns"]):
        dUs.append(mesh.increment(case, w[:, s]))
        ms.append(mesh.step(ms[-1], dUs[-1], tol))
    return ms, dUs


def _nll(case, u, y):
    return 0.5 * ((u[:, :: case["n"] // case["M"]] - y) / case["sigma"]).square().sum(-1)


def _exact_gradient(case, seed):
    m, dW, lam, y = (v.double() for v in _inputs(case, seed))
    mesh = _Mesh(case["n"])
    ms, dUs = _window(case, mesh, m, dW, lam, 1e-15)
    end = ms[-1].requires_grad_()
    nll = _nll(case, mesh.u(end), y)
    J = (nll + 0.5 * DT * lam.square().sum((1, 2))).detach()
    g = torch.autograd.grad(nll.sum(), end)[0]
    g_dW = torch.empty_like(dW)
    for s in reversed(range(case["Ns"])):
        m1, m0, dU = (v.detach().requires_grad_() for v in (ms[s + 1], ms[s], dUs[s]))
        R = mesh.residual(m1, m0, dU)
        psi = torch.zeros_like(g)
        for _ in range(300):      # J1^T psi = g, J1 = dR/dm1
            d = mesh.apply(1 / mesh.pic, g - torch.autograd.grad(R, m1, psi, retain_graph=True)[0])
            psi = psi + d
            if float(d.abs().max()) <= 1e-15 * float(psi.abs().max()):
                break
        g, g_dU = (-v for v in torch.autograd.grad(R, (m0, dU), psi))
        w = torch.zeros_like(dW[:, s]).requires_grad_()
        g_dW[:, s] = torch.autograd.grad(mesh.increment(case, w), w, g_dU)[0]
    return dict(J=J, g_m0=g, g_dW=g_dW, g_lam=DT * (g_dW + lam))


def _exact_net(case, params, u, y):
    """lambda [B, Ns, K] from 64-bit parameters."""
    n, K, Ns, C, M = case["n"], case["K"], case["Ns"], case["C"], case["M"]
    inn = torch.zeros_like(u)
    inn[:, :: n // M] = (y - u[:, :: n // M]) / case["sigma"]
    h, at, cin = torch.stack([u, inn], 1), 0, 2
    for _ in range(4):
        w = params[at:at + C * cin * 5].reshape(C, cin * 5)
        b = params[at + C * cin * 5:at + C * cin * 5 + C]
        at += C * cin * 5 + C
        Lo = h.shape[2] // 2
        tap = (2 * torch.arange(Lo, device="cuda")[:, None] + torch.arange(5, device="cuda") - 2) % h.shape[2]
        cols = h[:, :, tap].permute(0, 2, 1, 3).reshape(-1, cin * 5)
        h = torch.relu(cols @ w.T + b).reshape(-1, Lo, C).permute(0, 2, 1)
        cin = C
    P = n // 16
    ang = 2 * math.pi / P * torch.outer(torch.arange(P, dtype=torch.float64, device="cuda"),
                                        torch.arange(1, K // 2 + 1, dtype=torch.float64, device="cuda"))
    S = torch.stack([torch.sin(ang), torch.cos(ang)], 2).reshape(P, K) / P
    F = (h @ S).reshape(-1, C * K)
    Wh, bh = params[at:at + K * Ns * C * K].reshape(K * Ns, C * K), params[at + K * Ns * C * K:]
    return (F @ Wh.T + bh).reshape(-1, Ns, K)


def exact(case, seed):
    kind = case["kind"]
    if kind == "forecast":
        m, dW, lam, y = (None if v is None else v.double() for v in _inputs(case, seed))
        mesh = _Mesh(case["n"])
        ms, _ = _window(case, mesh, m, dW, lam, 1e-15 if case["dtype"] == "f64" else 1e-11)
        u = mesh.u(ms[-1])
        logG = torch.zeros(case["N"], dtype=torch.float64) if lam is None else \
            -(lam * dW + 0.5 * DT * lam.square()).sum((1, 2))
        return dict(m=ms[-1], u=u, nll=_nll(case, u, y), logG=logG, status=None)
    if kind == "gradient":
        return _exact_gradient(case, seed)
    if kind == "net":
        params, u, y, _, _ = _net_inputs(case, seed)
        return torch.cat([_exact_net(case, params.double(), v.double(), y.double()) for v in u.split(512)])
    if kind == "train":
        params, u, y, target, (m, v) = _net_inputs(case, seed)
        p = params.double().requires_grad_()
        loss = 0.0
        for ub, yb, tb in zip(u.double().split(256), y.double().split(256), target.double().split(256)):
            part = 0.5 / case["B"] * (_exact_net(case, p, ub, yb) - tb).square().sum()
            part.backward()
            loss = loss + part.detach()
        g, t = p.grad, 101
        m, v = 0.9 * m.double() + 0.1 * g, 0.999 * v.double() + 0.001 * g * g
        step = 1e-3 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
        return dict(loss=loss.reshape(1), grads=g, params=p.detach() - step, m=m, v=v)
    if kind == "weights":
        st = prepare(case, seed)
        phi, need = st["nll"] - st["logG"], case["ess"] * case["N"]

        def weights(d):
            w = torch.softmax(-d * phi, 0)
            return w, float(1 / w.square().sum())

        lo, hi, whole = 0.0, 1.0, weights(1.0)[1]
        if whole >= need:
            lo = 1.0
        else:
            for _ in range(60):
                mid = 0.5 * (lo + hi)
                lo, hi = (mid, hi) if weights(mid)[1] >= need else (lo, mid)
        w, e = weights(lo)
        return dict(wbar=w, out=torch.tensor([lo, e, lo, whole], dtype=torch.float64), idx=None, rows=[None] * 4)
    # cycles and the optimiser: their noise comes from the library's generator, and Metropolis decisions
    # and an optimiser's stop have no 64-bit value of their own
    return None
