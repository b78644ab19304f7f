"""FP64 steps by defect correction where the float side of an iteration ends: states so large
that the Helmholtz solve's right-hand side leaves the float range while m and its change stay
inside it (the time step is next to zero, so that the transport is the noise's alone and the step
is linear).  Such a step is run again by the plain FP64 iteration: m and u are the oracle's.
The conversions between the two sides over every exponent and scale: truncation, zero below the
float range, NaN above it.
"""
import ctypes
import subprocess

import numpy as np
import pytest
import torch

from paper_2402_06927_gb300 import build
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


@pytest.mark.parametrize("n", [128, 256])
def test_extreme_alpha_takes_the_plain_iteration(n):
    """alpha = 1e6 h, where the float Helmholtz solve is singular: a small launch gives what a large
    one does (the plain iteration on the same chunks), in the iterations of the oracle."""
    cfg = get_config("cfg1_f64", n=n)
    g, om = gpu_model(cfg, alpha=1e6 * cfg.h), oracle_model(cfg)
    N = 3 * torch.cuda.get_device_properties(0).multi_processor_count + 1
    m = tdev(np.stack([om.m_from_u(u) for u in random_state(cfg, 4, 3)]), g.dtype)
    dW = tdev(random_increments(cfg, 4, 4, steps=4), g.dtype)
    few = g.ensemble_step(m, dW)
    many = g.ensemble_step(m.repeat(-(-N // 4), 1), dW.repeat(-(-N // 4), 1, 1))
    torch.cuda.synchronize()
    for k in ("m", "u", "iters", "status"):
        assert torch.equal(few[k], many[k][:4]), k
    assert torch.all(few["status"] == 0) and torch.all(few["iters"] <= 4 * 4)


SOURCE = """
#include "sch_kernels.cuh"
__global__ void convert(int N, const double* x, const int* sh, unsigned* out, double* back) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const float f = sch::d2f_bits(x[i], sh[i] * (1 << 20));
    out[i] = __float_as_uint(f);
    back[i] = sch::f2d_bits(f, sh[i] * (1 << 20));
}
extern "C" void run(int N, const double* x, const int* sh, unsigned* out, double* back) {
    convert<<<(N + 255) / 256, 256>>>(N, x, sh, out, back);
}
"""


def test_scaled_conversions(tmp_path):
    src, so = tmp_path / "convert.cu", tmp_path / "convert.so"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", str(src), "-o", str(so)],
                   check=True, capture_output=True)
    r = np.random.default_rng(1)
    N = 200000
    e, sh = r.integers(0, 2048, N), r.integers(-1023, 801, N)
    sign, frac = r.integers(0, 2, N), r.integers(0, 1 << 52, N)
    bits = (sign << 63) | (e << 52) | frac
    x = torch.from_numpy(bits.astype(np.int64).view(np.float64).copy()).cuda()
    s = torch.from_numpy(sh.astype(np.int32)).cuda()
    out = torch.empty(N, dtype=torch.int32, device="cuda")
    back = torch.empty(N, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    ctypes.CDLL(str(so)).run(N, *[ctypes.c_void_p(t.data_ptr()) for t in (x, s, out, back)])
    torch.cuda.synchronize()
    inside = (e + sh >= 897) & (e + sh < 1151) & (e < 2047)
    ref = np.where(inside, (sign << 31) | ((e + sh - 896) << 23) | (frac >> 29), 0)
    ref = np.where((e == 2047) | (e + sh >= 1151), 0x7fffffff, ref)
    got = out.cpu().numpy().astype(np.int64) & 0xffffffff
    assert np.array_equal(got, ref)
    cut = ((bits >> 29) << 29).astype(np.int64).view(np.float64)
    assert np.array_equal(back.cpu().numpy()[inside], cut[inside])
