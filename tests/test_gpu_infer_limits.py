"""The convolutions' bounded waits running out (BF16 inference, 64 channels): a build of the pass
whose waits give up after a few tries.  Whatever the limit, the call returns, its output is either
the usual one or NaN throughout (NaN for certain when no wait is tried at all), and the device
goes on: the usual build gives the usual output afterwards in the same process.
"""
import os
import subprocess
import sys

import pytest

from paper_2402_06927_gb300 import build
from tests.helpers import require_lib

pytestmark = pytest.mark.gpu

SCRIPT = """
import sys
import torch
from paper_2402_06927_gb300 import _lib, api
g = torch.Generator(device="cpu").manual_seed(5)
u, y = torch.randn(%(B)d, 1024, generator=g).cuda(), torch.randn(64, generator=g).cuda()
def forward():
    net = api.ProposalNet(1024, 16, 20, 64, 0.05, seed=3, precision="bf16")
    out = [net.forward(u, y) for _ in range(3)]
    torch.cuda.synchronize()
    return out
usual_path = _lib.LIB_PATH
_lib.LIB_PATH = sys.argv[1]
cut = forward()
_lib.LIB_PATH, _lib._LIB = usual_path, None
usual = forward()
assert torch.all(torch.isfinite(usual[0])) and all(torch.equal(usual[0], o) for o in usual)
nan = [bool(torch.all(torch.isnan(o))) for o in cut]
assert all(n or torch.equal(o, usual[0]) for n, o in zip(nan, cut))
print("NAN" if all(nan) else "MIXED")
"""


@pytest.mark.parametrize("limit", [0, 1, 3, 40])
def test_waits_that_run_out_give_nan(limit, tmp_path):
    require_lib()
    obj, lib = str(tmp_path / "nn_infer.o"), str(tmp_path / "libcut.so")
    run = lambda *a: subprocess.run(a, check=True, capture_output=True)  # noqa: E731
    run(build.nvcc(), *build.ARCH, *build.FLAGS, f"-DSCH_CONV_WAIT_LIMIT={limit}", "-c",
        os.path.join(build.CSRC, "nn_infer.cu"), "-o", obj)
    others = [os.path.join(build.BUILD, os.path.basename(s).replace(".cu", ".o")) for s in build.sources()
              if os.path.basename(s) != "nn_infer.cu"]
    run(build.nvcc(), *build.ARCH, "-shared", "-o", lib, obj, *others, "-lcudart")
    for B in (2, 700):
        r = subprocess.run([sys.executable, "-c", SCRIPT % dict(B=B), lib], capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr[-2000:]
        assert r.stdout.strip() == "NAN" or limit > 0
