"""Runs on both sides of the lengths from which one launch takes all steps: the
stresses are those of stepping bitwise, and the gradients those of the oracle (2e-4
normwise, the FP32 gradients' bound) from the trajectory and from checkpoints
one, two and three steps apart, whose last segment may be shorter."""
import numpy as np
import pytest

from helpers import ensure_lib
from oracle import orc
from test_gpu_run import oracle_problem, problem, solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,m", [(2, (9, 5), 5), (2, (7, 5), 49), (3, (5, 4, 3), 7), (3, (4, 3, 3), 8), (3, (5, 3, 2), 16)])
@pytest.mark.parametrize("steps", [1, 2, 3, 7, 8])
def test_run_and_gradients(dim, n, m, steps):
    import torch
    ensure_lib()
    case, kap, u, sigma0, lam = problem(dim, n, m, steps, False)
    ref = orc.gradients(oracle_problem(case), sigma0, kap, u, steps, lam)
    s = solver(case, 1)
    t = lambda a: torch.as_tensor(a, dtype=s.dtype, device="cuda").contiguous()
    kt = t(kap)
    s.set_state(t(sigma0))
    rows = s.run(steps, kt)
    grads = [s.backward_run(t(lam), rows, kt)]
    for K in (1, 2, 3):
        s.set_state(t(sigma0))
        ckpts = []
        for k in range(steps):
            if k % K == 0:
                ckpts.append(s.new_checkpoint())
                s.save(ckpts[-1])
            s.step(kt, kt)
            assert torch.equal(rows[k], s.stress()), k
        grads.append(s.backward(t(lam), ckpts, K, steps, kt))
        assert s.step_index() == min(K, steps)     # the state after the first segment, recomputed last
        assert torch.equal(rows[min(K, steps) - 1], s.stress())
    s.close()
    for g in grads:
        for got, want in ((g[0].cpu().numpy(), ref["sigma0"]), (g[1].cpu().numpy(), ref["kappa"]),
                          (np.array([g[2]]), np.array([ref["Wi"]])), (np.array([g[3]]), np.array([ref["beta"]]))):
            assert np.max(np.abs(got - want)) < 2e-4 * np.max(np.abs(want))


@pytest.mark.parametrize("dim,n", [(2, (9, 5)), (3, (5, 4, 3))])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_infinite_gradients_as_in_single_steps(dim, n, value):
    # kappa* = 2 kappa - kappa of an infinite kappa is not a number: the point's stresses and gradients are none
    import torch
    ensure_lib()
    steps = 9
    case, kap, u, sigma0, lam = problem(dim, n, 8, steps, False)
    kap[0, 7] = value
    s = solver(case, 1)
    t = lambda a: torch.as_tensor(a, dtype=s.dtype, device="cuda").contiguous()
    kt = t(kap)
    s.set_state(t(sigma0))
    rows = s.run(steps, kt)
    whole = s.backward_run(t(lam), rows, kt)
    s.set_state(t(sigma0))
    ckpts = []
    for k in range(steps):
        ckpts.append(s.new_checkpoint())
        s.save(ckpts[-1])
        s.step(kt, kt)
        assert torch.equal(torch.isnan(rows[k]), torch.isnan(s.stress()))
    single = s.backward(t(lam), ckpts, 1, steps, kt)
    s.close()
    for a, b in zip(whole[:2], single[:2]):
        assert torch.equal(torch.isnan(a), torch.isnan(b))
        assert torch.isnan(b[:, 7]).any() and torch.isfinite(b[:, 8]).all()
