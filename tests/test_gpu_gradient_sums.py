"""The gradients of FP32 storage are accumulated in FP64.

Runs of one launch against the same reverse sweep by twos (checkpoints at every second step: the
same adjoint values in FP32, the contributions of two steps at a time added to the FP64
fields).  At most 1e-13 of the largest entry: 200 FP64 additions of either order,
also where the values are near the lower end of the FP32 range (dJ scaled by
2^-112), at which a float's rounding error is no longer representable, and at the
upper end (2^112, and 2^54 with stresses of 2^70, whose products with lamR leave it
before dt is applied; dJ/dWi and dJ/dbeta, FP32 sums per point, then do as well)."""
import numpy as np
import pytest

from helpers import ensure_lib
from test_gpu_run import problem, solver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


@pytest.mark.parametrize("dim,n,m", [(2, (43, 3), 8), (2, (8, 4), 33), (3, (5, 4, 3), 24)])
@pytest.mark.parametrize("exponent,stretch", [(0, 0), (-112, 0), (112, 0), (54, 70)])
def test_runs_accumulate_in_fp64(dim, n, m, exponent, stretch):
    import torch
    steps = 150
    case, kap, u, sigma0, lam = problem(dim, n, m, steps, False)
    sigma0 = np.ldexp(sigma0, stretch)
    s = solver(case, 1)
    t = lambda a: torch.as_tensor(a, dtype=s.dtype, device="cuda").contiguous()
    kt, dJ = t(kap), t(np.ldexp(lam, exponent))
    s.set_state(t(sigma0))
    got = s.backward_run(dJ, s.run(steps, kt), kt)
    s.set_state(t(sigma0))
    ckpts = []
    for k in range(steps):
        if k % 2 == 0:
            ckpts.append(s.new_checkpoint())
            s.save(ckpts[-1])
        s.step(kt, kt)
    ref = s.backward(dJ, ckpts, 2, steps, kt)
    s.close()
    for a, b in list(zip(got, ref))[:2 if stretch else 4]:
        a, b = (np.asarray(v.cpu().numpy() if hasattr(v, "cpu") else v) for v in (a, b))
        assert np.all(np.isfinite(b))
        assert np.max(np.abs(a - b)) <= 1e-13 * np.max(np.abs(b))
