"""What the calls of whole runs record, refuse and touch."""
import numpy as np
import pytest

from helpers import ensure_lib
from test_gpu_run import problem, solver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def make(precision=1, transport=False):
    import torch
    case, kap, u, sigma0, lam = problem(2, (40, 24), 8, 40, transport)
    s = solver(case, precision)
    t = lambda a: torch.as_tensor(a, dtype=s.dtype, device="cuda").contiguous()
    return s, t(kap), t(u) if transport else None, t(sigma0), t(lam)


@pytest.mark.parametrize("precision,steps", [(1, 40), (1, 1), (0, 3)])
def test_events_are_recorded_by_a_run(precision, steps):
    import torch
    s, kt, _, sigma0, _ = make(precision)
    before, after, start = (torch.cuda.Event(enable_timing=True) for _ in range(3))
    before.record()
    after.record()
    torch.cuda._sleep(100000)
    start.record()
    s.set_state(sigma0)
    s.set_step_events(before, after)
    s.run(steps, kt)
    s.set_step_events(None, None)
    torch.cuda.synchronize()
    assert start.elapsed_time(before) >= 0.0
    assert before.elapsed_time(after) > 0.0
    s.close()
