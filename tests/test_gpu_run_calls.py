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


def test_refusals_of_the_reverse_run():
    import torch
    from paper_2411_17294_gb300 import tfs

    def code(f):
        with pytest.raises(tfs.TfsError) as err:
            f()
        return err.value.code

    s, kt, _, sigma0, lam = make()
    traj = torch.zeros((2, 3, s.N), dtype=s.dtype, device="cuda")
    assert code(lambda: s.backward_run(lam, traj, kt)) == tfs.TFS_ERR_STATE       # no state set
    s.close()
    case = problem(2, (40, 24), 8, 1, False)[0]
    s = tfs.Solver(2, (40, 24), 0.5, 1.3, 0.4, 2e-3, m=8, precision=1, transport=False)
    s.set_state(sigma0)
    assert code(lambda: s.backward_run(lam, traj, kt)) == tfs.TFS_ERR_NOSOE       # no table
    s.set_soe(case["mu"], case["w"])
    s.backward_run(lam, s.run(2, kt), kt)
    s.close()


def test_trajectory_of_another_stream():
    # a block of the trajectory's size, freed on the current stream with a write to it still pending there
    import torch
    s, kt, _, sigma0, _ = make()
    s.set_state(sigma0)
    ref = s.run(40, kt)
    s.set_state(sigma0)
    side = torch.cuda.Stream()
    block = torch.empty_like(ref)
    torch.cuda.synchronize()
    torch.cuda._sleep(50000000)
    block.fill_(7.0)
    del block
    got = s.run(40, kt, stream=side)
    torch.cuda.synchronize()
    assert torch.equal(got, ref)
    s.close()
