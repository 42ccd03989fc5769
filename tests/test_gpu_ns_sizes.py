"""The velocity step at the edges of its row passes, against the NumPy oracle: the
shortest and longest rows, rows that fill a block alone or by the hundred,
lengths with and without a last radix-2 stage, with and without a stress and a
previous level.  1e-12 normwise, as the step's other comparisons (both sides FP64)."""
import numpy as np
import pytest

from helpers import ensure_lib, rel_err_per_component
from oracle.ns import NSOracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


@pytest.mark.parametrize("n", [(2, 2), (2, 8), (1024, 2), (2, 1024), (4, 16), (8, 512), (128, 32), (256, 1024)])
@pytest.mark.parametrize("stress,past", [(True, False), (False, True), (True, True)])
def test_step_matches_oracle(n, stress, past):
    import torch
    from paper_2411_17294_gb300 import tfs
    L, beta, Re, dt = (2.0, 3.0), 0.6, 20.0, 5e-3
    rng = np.random.default_rng(n[0] + 3 * n[1])
    N = n[0] * n[1]
    u0, up = rng.normal(size=(2, N)), rng.normal(size=(2, N))
    o = NSOracle(n, L, beta, Re, dt)
    o.set_state(u0, up if past else None)
    s = tfs.NSSolver(n, L, beta, Re, dt, precision=tfs.TFS_FP64)
    s.set_state(u0, up if past else None)
    for _ in range(3):
        sg = rng.normal(size=(3, N)) if stress else None
        u_ref, k_ref = o.step(sg)
        u, k = s.step(torch.as_tensor(sg, device="cuda") if stress else None)
    s.close()
    assert np.all(rel_err_per_component(u.cpu().numpy(), u_ref) < 1e-12)
    scale = np.max(np.abs(k_ref))      # a component may vanish identically (axes of two points)
    assert np.max(np.abs(k.cpu().numpy() - k_ref)) <= 1e-12 * max(scale, 1e-300)
