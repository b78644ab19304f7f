"""The BF16 inference pass (64 channels, n a multiple of 1024) at its awkward sizes: a lone sample, a
batch past one tile per SM, layers of one 64-row tile, of whole 128-row tiles and of 64-row tiles
at three quarters of a power of two, odd and large mode counts, drift counts off the head's tile.

A sample's lambda does not depend on the batch it is in: every contraction runs over the
sample's own k-order whatever the tile, so a batch equals its samples bit for bit.  A
sample by itself is held to the oracle with BF16 operands (2e-3, as the other BF16 tests).
"""
import numpy as np
import pytest
import torch

from oracle import convnet as CN
from tests.helpers import require_lib
from tests.test_gpu_proposal import _case, _flat

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1024, 16, 20, 64, 700), (1024, 7, 3, 64, 3), (1024, 66, 2, 64, 2),
                                   (2048, 8, 7, 128, 90), (3072, 6, 13, 96, 5), (4096, 32, 10, 128, 33)])
def test_batch_equals_its_samples(shape):
    api = require_lib()
    n, K, Ns, M, B = shape
    p, u, y, _ = _case(n, K, Ns, 64, M, B=B, seed=21)
    y[:, 5] = np.nan
    net = api.ProposalNet(n, K, Ns, M, 0.05, C=64, params=torch.tensor(_flat(p), dtype=torch.float32),
                          precision="bf16")
    ud = torch.tensor(u, dtype=torch.float32, device="cuda")
    yd = torch.tensor(y, dtype=torch.float32, device="cuda")
    lam = net.forward(ud, yd)
    shared = net.forward(ud, yd[0].contiguous())
    torch.cuda.synchronize()
    assert torch.all(torch.isfinite(lam))
    for b in sorted({0, 1, B // 2, B - 1}):
        one = net.forward(ud[b:b + 1].contiguous(), yd[b:b + 1].contiguous())
        assert torch.equal(one[0], lam[b])
        assert torch.equal(net.forward(ud[b:b + 1].contiguous(), yd[0].contiguous())[0], shared[b])
    if K % 2:   # the interface's K counts sin/cos pairs, and so does the oracle's mode table
        return
    x0 = CN.features(u[:1], y[0], 0.05)
    ref, _ = CN.forward(p, x0, K, Ns, operands="bf16")
    assert np.max(np.abs(lam[:1].cpu().numpy() - ref)) <= 2e-3 * np.max(np.abs(ref))
