"""Branches taken by size or by caller, each against the general form:

* tempering: the float location of the root and its FP64 Newton finish, at dead particles
  (infinite phi), two-valued phi, roots many octaves below the remaining step, and
  particle counts at the edges of a thread's share.
"""
import numpy as np
import pytest
import torch

from oracle import filter as OF
from paper_2402_06927_gb300 import api
from tests.helpers import tdev

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
