"""The paper's variable with a table whose weights are all zero (accepted by
tfs_set_soe): Psi = xi Phi + h = 0 at every step, in both storage forms; Phi
follows its own equation without dividing by xi = 0."""
import numpy as np
import pytest

from helpers import ensure_lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n", [(2, (9, 5)), (3, (5, 4, 3))])
def test_stress_is_zero(dim, n):
    import torch
    ensure_lib()
    from paper_2411_17294_gb300 import tfs
    rng = np.random.default_rng(4)
    N, nc = int(np.prod(n)), 3 if dim == 2 else 6
    kap, sigma0 = (rng.normal(size=(k, N)) for k in (dim * dim, nc))
    phi = []
    for precision in (0, 1):
        s = tfs.Solver(dim, n, 0.5, 1.3, 0.4, 1e-2, m=3, precision=precision, mu=np.array([0.5, 4.0, 30.0]),
                       w=np.zeros(3), transport=False, form="paper")
        t = lambda a: torch.as_tensor(a, dtype=s.dtype, device="cuda").contiguous()
        s.set_state(t(sigma0))
        kt = t(kap)
        for _ in range(3):
            s.step(kt, kt)
        assert torch.all(s.stress() == 0.0)
        assert s.status() == 0
        buf = s.new_checkpoint()
        s.save(buf)
        phi.append(buf[256:256 + nc * N * (8 if precision == 0 else 4)].view(s.dtype).double().cpu().numpy())
        s.close()
    # without Psi the right-hand sides are -b1 Phi^n - b2 Phi^{n-1}: Phi stays Phi^0
    for got, tol in zip(phi, (1e-14, 1e-6)):
        assert np.max(np.abs(got.reshape(nc, N) - sigma0)) < tol * 10
