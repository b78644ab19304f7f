"""The host's share of a filter cycle: a cycle of one stage is a few library calls, an event and the
copy of the stages' results, and dispatches no other tensor operation."""
import numpy as np
import pytest
import torch
from torch.utils._python_dispatch import TorchDispatchMode

from paper_2402_06927_gb300.filter import EnsembleFilter
from workloads import get_config, random_obs, random_state
from tests.helpers import gpu_model, oracle_model, tdev

pytestmark = pytest.mark.gpu


class _Ops(TorchDispatchMode):
    def __init__(self):
        super().__init__()
        self.names = []

    def __torch_dispatch__(self, func, types, args=(), kwargs=None):
        self.names.append(func.overloadpacket.__name__)
        return func(*args, **(kwargs or {}))


def test_one_stage_cycle_dispatches_one_copy():
    cfg = get_config("cfg2_f32", n=256, sigma=5.0, M=16)
    g, om = gpu_model(cfg), oracle_model(cfg)
    f = EnsembleFilter(g, 24, 4, 12.0, 0.99, 2, 3)
    f.set_state(tdev(np.stack([om.m_from_u(u) for u in random_state(cfg, 24, 3)]), g.dtype))
    y = tdev(random_obs(cfg, 8), g.dtype)
    f.cycle(y, 0)
    with _Ops() as ops:
        st = f.cycle(y, 1)
    assert len(st.stages) == 1
    assert ops.names == ["copy_"]


def test_given_outputs_are_checked():
    """ensemble_step checks the outputs that a caller gives, each by shape, type and layout."""
    cfg = get_config("cfg2_f32", n=256, M=16)
    g = gpu_model(cfg)
    m, dW = torch.zeros(3, 256, device="cuda"), torch.zeros(3, 2, g.K, device="cuda")
    y = torch.zeros(16, device="cuda")
    for name, good in (("m_out", m), ("u_out", m), ("nll", m[:, 0].double()), ("logG", m[:, 0].double())):
        g.ensemble_step(m, dW, None, y, **{name: torch.empty_like(good)})
        for bad in (torch.empty_like(good)[:2], torch.empty_like(good).half(), torch.empty_like(good).cpu(),
                    torch.empty((2 * g.n, 3), device="cuda", dtype=good.dtype).t()[:, ::2].squeeze()):
            with pytest.raises((TypeError, ValueError)):
                g.ensemble_step(m, dW, None, y, **{name: bad})


def test_calls_run_on_the_current_stream():
    """The stream handed to the library is torch's current one: of the context, else the default."""
    from paper_2402_06927_gb300 import api
    s = torch.cuda.Stream()
    assert api._stream() == torch.cuda.current_stream().cuda_stream
    with torch.cuda.stream(s):
        assert api._stream() == s.cuda_stream
    assert api._stream(s) == s.cuda_stream
    assert api._stream() == torch.cuda.current_stream().cuda_stream
