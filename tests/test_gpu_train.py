"""The BF16 training pass on channels-first activations (64 channels) at its awkward sizes:
layers shorter than a tile (several samples in one), tiles that end past the batch, drift
counts that are no multiple of the copies' width, k-chunks that start off a 16-byte boundary.

A batch of B = 2^k samples must give the mean of its samples' own gradients: the loss
gradient's 1/B is an exact scale, so every BF16 operand of a sample is the same (scaled) value
in both, and only FP32 sums are ordered differently.  A weight gradient's sum runs
through at most about 40 tensor-core steps a chunk and 512 chunks, and the samples' mean adds
at most 64 terms: at most 2^10 roundings of 2^-24 on sums that the samples' largest entries
bound, so 2^-14 of their mean.  A sample by itself is held to the oracle with BF16 operands.
"""
import numpy as np
import pytest
import torch

from oracle import convnet as CN
from tests.helpers import require_lib
from tests.test_gpu_proposal import _case, _flat, _unflat

pytestmark = pytest.mark.gpu

SHAPES = [(128, 2, 1, 8, 1), (128, 6, 3, 32, 2), (128, 6, 3, 32, 64), (256, 4, 5, 16, 16), (512, 20, 9, 32, 8),
          (1024, 6, 13, 64, 4), (1024, 16, 20, 64, 64), (2048, 8, 7, 128, 2)]


def _net(shape, seed):
    api = require_lib()
    n, K, Ns, M, B = shape
    p, u, y, target = _case(n, K, Ns, 64, M, B=B, seed=seed)
    y[:, 3] = np.nan
    net = api.ProposalNet(n, K, Ns, M, 0.05, C=64, params=torch.tensor(_flat(p), dtype=torch.float32),
                          precision="bf16")
    dev = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")
    return net, p, (dev(u), dev(y), dev(target)), (u, y, target)


@pytest.mark.parametrize("shape", SHAPES)
def test_batch_gradient_is_the_samples_mean(shape):
    net, p, (u, y, t), _ = _net(shape, 11)
    B = shape[4]
    loss, grads = net.loss_and_grad(u, y, t)
    again = net.loss_and_grad(u, y, t)[1]
    assert torch.equal(grads, again)
    mean, size, Ls = None, 0.0, 0.0
    parts = [net.loss_and_grad(u[b:b + 1].contiguous(), y[b:b + 1].contiguous(), t[b:b + 1].contiguous())
             for b in range(B)]
    split = lambda g: _unflat(g.cpu().numpy().astype(np.float64), p)
    gs = [split(g) for _, g in parts]
    full = split(grads)
    for k in full:
        mean = sum(g[k] for g in gs) / B
        size = sum(np.max(np.abs(g[k])) for g in gs) / B
        assert np.max(np.abs(full[k] - mean)) <= 2.0 ** -14 * size, k
    Ls = sum(l.item() for l, _ in parts) / B
    assert abs(loss.item() - Ls) <= 1e-5 * Ls


@pytest.mark.parametrize("shape", [(128, 2, 1, 8, 1), (512, 20, 9, 32, 1), (2048, 8, 7, 128, 1)])
def test_one_sample_matches_oracle(shape):
    net, p, (u, y, t), (u0, y0, t0) = _net(shape, 12)
    n, K, Ns, M, B = shape
    x0 = CN.features(u0, y0[0], 0.05)
    L, g = CN.loss_and_grad(p, x0, t0, K, Ns, operands="bf16")
    loss, grads = net.loss_and_grad(u, y, t)
    assert abs(loss.item() - L) <= 2e-3 * L
    gg = _unflat(grads.cpu().numpy().astype(np.float64), p)
    for k in g:   # a flipped ReLU mask or BF16 neighbour moves one sample's gradient by more than a batch's
        assert np.linalg.norm(gg[k] - g[k]) <= 5e-2 * np.linalg.norm(g[k]), k
