"""FP64 point systems whose numbers leave the range of the FP32 factors or of a
scaled FP32 vector: the matrix (relaxation below 1e-38, velocity gradients
above 1e38, both sides of the float limit) and components of one point far apart.
Against the FP64 oracle, pointwise at the bounds of the ordinary systems (1e-11
forward, 1e-9 reverse); components of decoupled systems each at that bound."""
import numpy as np
import pytest

from helpers import ensure_lib, run_gpu, run_oracle
from test_gpu_fp64_step import fields, table

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def system(dim, n, kind):
    alpha, dt, m = 0.5, 1e-2, 6
    mu, w = table(alpha, dt, m)
    _, kap, sigma0 = fields(dim, n, 3)
    N, Wi = kap.shape[1], 0.9
    rng = np.random.default_rng(8)
    if kind == "relaxation":                 # a = eta + dt/Wi = 1e43
        Wi = 1e-45
    elif kind == "edge":                     # a just inside the float range: its reciprocal is subnormal
        Wi = dt / 3e38
    elif kind == "gradient":                 # one huge diagonal entry, in some points of each tile
        kap[0] = np.where(rng.random(N) < 0.3, -1e45, kap[0])
        kap[1:] *= 1e-3
    elif kind == "apart":                    # components from 1 to 1e-60 at one point, no coupling
        kap = np.zeros_like(kap)
        sigma0 = sigma0 * 10.0 ** (-12.0 * np.arange(len(sigma0)))[:, None]
    return dict(dim=dim, n=n, alpha=alpha, Wi=Wi, beta=0.5, dt=dt, mu=mu, w=w), kap, sigma0


KINDS = ["relaxation", "edge", "gradient", "apart"]


@pytest.mark.parametrize("dim,n", [(2, (40, 3)), (3, (9, 4, 3))])
@pytest.mark.parametrize("kind", KINDS)
def test_step(dim, n, kind):
    case, kap, sigma0 = system(dim, n, kind)
    if kind == "apart" and dim == 2:
        sigma0[2] *= 1e-30
    got = run_gpu(case, sigma0, kap, None, 1, 0)
    ref = run_oracle(case, sigma0, kap, None, 1)
    assert np.all(np.isfinite(ref)) and np.any(ref != 0.0)
    scale = np.abs(ref) if kind == "apart" else np.max(np.abs(ref), axis=0)
    assert np.all(np.abs(got - ref) <= 1e-11 * scale)


@pytest.mark.parametrize("dim,n", [(2, (40, 3)), (3, (9, 4, 3))])
@pytest.mark.parametrize("kind", KINDS)
def test_reverse_step(dim, n, kind):
    import torch
    from oracle import orc
    from paper_2411_17294_gb300 import tfs
    case, kap, sigma0 = system(dim, n, kind)
    lam = np.random.default_rng(9).normal(size=sigma0.shape)
    if kind == "apart":
        lam = lam * 10.0 ** (-12.0 * np.arange(len(lam)))[:, None]
        if dim == 2:
            lam[2] *= 1e-30
    ref = orc.gradients(orc.Problem(**case), sigma0, kap, None, 1, lam)
    s = tfs.Solver(dim, n, case["alpha"], case["Wi"], case["beta"], case["dt"], m=len(case["mu"]),
                   precision=tfs.TFS_FP64, mu=case["mu"], w=case["w"], transport=False)
    t = lambda a: torch.as_tensor(a, dtype=torch.float64, device="cuda").contiguous()
    s.set_state(t(sigma0))
    kt = t(kap)
    g = s.backward_run(t(lam), s.run(1, kt), kt)
    s.close()
    got, want = g[0].cpu().numpy(), ref["sigma0"]
    assert np.any(want != 0.0)
    scale = np.abs(want) if kind == "apart" else np.max(np.abs(want), axis=0)
    assert np.all(np.abs(got - want) <= 1e-9 * scale)
    got, want = g[1].cpu().numpy(), ref["kappa"]
    assert np.all(np.abs(got - want) <= 1e-9 * np.max(np.abs(want), axis=0))
