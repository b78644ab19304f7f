"""Tempering where the ESS is nearly flat at its threshold: a tight cluster of particles whose
number is just above ess_min and a far one, so that the ESS stays within 1e-9 of ess_min over
decades of dtheta and the slope of the search's Newton steps drowns in rounding.

The answer is the largest passing dtheta to a relative 2^-49 or within a bracket as narrow, so
the ESS there is ess_min but for the rounding of the kernel's sums.  Its bound: a weight of the
cluster is exp(-x), x < 1e-3, right to 2^-52; the sums S1 and S2 take at most eight additions a
thread, five in the warp and six over the cluster of CTAs, 19 x 2^-53 relative; ESS = S1^2 / S2 then
holds 3 (19 x 2^-53 + 2^-52) = 7e-15, and the bracket's width moves it by less than 1e-3 x 2^-49.
"""
import numpy as np
import pytest
import torch

from paper_2402_06927_gb300 import api
from tests.helpers import tdev

pytestmark = pytest.mark.gpu


def _two_clusters(seed):
    r = np.random.default_rng(seed)
    n1, n2 = int(r.integers(2, 600)), int(r.integers(1, 600))
    phi = np.concatenate([r.random(n1) * 10 ** r.uniform(-6, -3), 10 ** r.uniform(3, 7) + r.gamma(2.0, 5.0, n2)])
    return phi, n1 * (1 - 10 ** r.uniform(-12, -9))


def _ess(phi, d):
    w = np.exp(-np.longdouble(d) * (phi.astype(np.longdouble) - np.longdouble(phi.min())))
    return w.sum() ** 2 / (w * w).sum()


def test_flat_ess_is_searched_to_its_root():
    cases = [_two_clusters(k) for k in range(600)]
    outs = [api.pf_temper(tdev(phi, torch.float64), None, 0.0, ess)[1] for phi, ess in cases]
    torch.cuda.synchronize()
    searched = 0
    for (phi, ess), out in zip(cases, outs):
        d = out[0].item()
        if d < 1.0:
            searched += 1
            assert abs(float(_ess(phi, d) / np.longdouble(ess) - 1)) <= 1e-14
    assert searched > 100
