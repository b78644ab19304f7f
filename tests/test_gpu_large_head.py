"""A head of more than 2^31 entries (64 modes, 8200 steps, 64 channels: 8.6 GB of weights) in BF16:
the passes of 64 channels count the head's entries in 32 bits and leave it to the generic one.

Forward and weight gradients against the same network with FP32 operands: BF16 operands are right to
2^-9, five roundings one after the other (four layers, the mode features) and the head's own make
6 x 2^-9 = 1.2e-2 in norm at the worst.
"""
import pytest
import torch

from tests.helpers import require_lib

pytestmark = pytest.mark.gpu


def test_head_beyond_32_bits():
    api = require_lib()
    n, K, Ns, M, B = 1024, 64, 8200, 64, 2
    g = torch.Generator(device="cuda").manual_seed(3)
    conv = 64 * 2 * 5 + 64 + 3 * (64 * 64 * 5 + 64)
    head = K * Ns * 64 * K
    assert head > 2 ** 31
    params = torch.empty(conv + head + K * Ns, device="cuda")
    params[:conv].normal_(0.0, 0.08, generator=g)
    params[conv:].normal_(0.0, 1 / 64, generator=g)
    u = 0.3 * torch.randn(B, n, generator=g, device="cuda")
    y = 0.3 * torch.randn(M, generator=g, device="cuda")
    target = 0.1 * torch.randn(B, Ns, K, generator=g, device="cuda")
    net = api.ProposalNet(n, K, Ns, M, 0.5, C=64, params=params, precision="bf16")
    lam = net.forward(u, y)
    loss, grads = net.loss_and_grad(u, y, target)
    net.set_precision("fp32")
    ref = net.forward(u, y)
    assert float((lam - ref).norm()) <= 1.2e-2 * float(ref.norm())
    rl, rg = net.loss_and_grad(u, y, target)
    assert abs(float(loss) - float(rl)) <= 2.5e-2 * float(rl)
    for part in (slice(conv, conv + head // 2), slice(conv + head // 2, conv + head), slice(conv + head, None)):
        assert float((grads[part] - rg[part]).norm()) <= 2.5e-2 * float(rg[part].norm())
