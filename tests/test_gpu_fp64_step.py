"""The FP64 step kernel at the sizes where it can go wrong, against the FP64
oracle at the FP64 mode's bound (1e-11 normwise): tiles that end past the grid,
numbers of modes around the load-ahead depth and the largest table, tile counts
on both sides of the split of a tile's modes, grids shorter than the stencil,
and point systems that the FP32-factored refinement cannot take (ill
conditioned, outside the FP32 range), which go to FP64 elimination."""
import numpy as np
import pytest

from helpers import ensure_lib, rel_err_per_component, run_gpu, run_oracle, stable_velocity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def table(alpha, dt, m):
    """m geometric exponents with the weights of the trapezoidal rule in log mu."""
    mu = np.geomspace(0.1, 2.0 / dt, m) if m > 1 else np.array([1.0])
    h = np.log(mu[1] / mu[0]) if m > 1 else 1.0
    return mu, h * np.sin(np.pi * alpha) / np.pi * mu ** alpha


def fields(dim, n, seed):
    rng = np.random.default_rng(seed)
    N = int(np.prod(n))
    return rng.normal(size=(dim, N)), rng.normal(size=(dim * dim, N)), rng.normal(size=(3 if dim == 2 else 6, N))


@pytest.mark.parametrize("dim,n,m,alpha,stencil,eps", [
    (2, (1, 1), 1, 0.5, 0, 0.0), (2, (3, 2), 7, 0.5, 0, 0.0), (2, (31, 1), 8, 0.5, 1, 0.0),
    (2, (33, 1), 9, 0.3, 0, 1e-4), (2, (40, 37), 33, 0.7, 0, 0.0), (2, (8, 4), 64, 0.5, 1, 1e-4),
    (2, (97, 101), 16, 0.5, 0, 0.0), (2, (98, 101), 17, 0.5, 0, 1e-5), (2, (12, 8), 0, 1.0, 0, 0.0),
    (3, (2, 1, 3), 5, 0.5, 0, 0.0), (3, (5, 4, 3), 8, 0.6, 1, 1e-3), (3, (16, 2, 1), 64, 0.4, 0, 0.0),
    (3, (21, 21, 22), 6, 0.5, 0, 0.0), (3, (23, 21, 22), 11, 0.5, 0, 1e-4), (3, (7, 6, 5), 0, 1.0, 1, 0.0)])
@pytest.mark.parametrize("transport", [False, True])
def test_step_matches_oracle(dim, n, m, alpha, stencil, eps, transport):
    dt, steps = 2e-3, 4
    mu, w = table(alpha, dt, m) if m else (np.zeros(0), np.zeros(0))
    u, kap, sigma0 = fields(dim, n, 7 + m)
    case = dict(dim=dim, n=n, alpha=alpha, Wi=1.3, beta=0.4, dt=dt, stencil=stencil, eps=eps if transport else 0.0,
                transport=transport)
    if m:
        case.update(mu=mu, w=w)
    if transport:
        u = stable_velocity(case, u, 0.5)
    seq = lambda k: kap * (1.0 + 0.1 * k)
    got = run_gpu(case, sigma0, seq, u, steps, 0)
    ref = run_oracle(case, sigma0, seq, u, steps)
    assert np.all(rel_err_per_component(got, ref) < 1e-11)


@pytest.mark.parametrize("dim,n", [(2, (40, 3)), (3, (9, 4, 3))])
@pytest.mark.parametrize("kind", ["indefinite", "mixed", "tiny", "huge", "zero"])
def test_systems_beyond_the_refinement(dim, n, kind):
    # indefinite: dt |kappa| far above the diagonal; mixed: such points scattered among ordinary ones
    # of the same tiles; tiny and huge: stresses and sources outside the FP32 range (1e-150, 1e150);
    # zero: no source at all on half of the points
    alpha, dt, m = 0.5, 1e-2, 6
    mu, w = table(alpha, dt, m)
    _, kap, sigma0 = fields(dim, n, 3)
    rng = np.random.default_rng(5)
    N = int(np.prod(n))
    if kind == "indefinite":
        kap = kap * 300.0
    elif kind == "mixed":
        kap = kap * np.where(rng.random(N) < 0.2, 300.0, 0.5)
    elif kind in ("tiny", "huge"):
        sigma0 = sigma0 * (1e-150 if kind == "tiny" else 1e150)
        kap = kap * 1e-3 if kind == "huge" else np.zeros_like(kap)
    else:
        on = rng.random(N) < 0.5
        kap, sigma0 = kap * on, sigma0 * on
    case = dict(dim=dim, n=n, alpha=alpha, Wi=0.9, beta=0.5, dt=dt, mu=mu, w=w)
    got = run_gpu(case, sigma0, kap, None, 2, 0)
    ref = run_oracle(case, sigma0, kap, None, 2)
    assert np.all(np.isfinite(got))
    # pointwise: elimination and refinement both solve to a few ulp of the point's own norm times its
    # condition (up to about 1e5 among these matrices)
    scale = np.max(np.abs(ref), axis=0)
    assert np.max(np.max(np.abs(got - ref), axis=0)[scale > 0] / scale[scale > 0]) < 1e-11
    assert np.all(got[:, scale == 0] == 0.0)


@pytest.mark.parametrize("dim,n", [(2, (40, 3)), (3, (9, 4, 3))])
@pytest.mark.parametrize("scale", [0.5, 300.0])
def test_adjoint_of_ordinary_and_indefinite_systems(dim, n, scale):
    # the transposed point systems through the same refinement and elimination; two steps from a random
    # stress, every entry of the gradients against the oracle's reverse sweep.  1e-9 of the largest: two reverse steps
    # through systems of condition up to 1e5.
    import torch
    from oracle import orc
    from paper_2411_17294_gb300 import tfs
    alpha, dt, m, steps = 0.5, 1e-2, 6, 2
    mu, w = table(alpha, dt, m)
    _, kap, sigma0 = fields(dim, n, 3)
    kap = kap * scale
    lam = np.random.default_rng(9).normal(size=sigma0.shape)
    prob = orc.Problem(dim=dim, n=n, alpha=alpha, Wi=0.9, beta=0.5, dt=dt, mu=mu, w=w)
    ref = orc.gradients(prob, sigma0, kap, None, steps, lam)
    s = tfs.Solver(dim, n, alpha, 0.9, 0.5, dt, m=m, precision=tfs.TFS_FP64, mu=mu, w=w, transport=False)
    t = lambda a: torch.as_tensor(a, dtype=torch.float64, device="cuda").contiguous()
    s.set_state(t(sigma0))
    kt = t(kap)
    g = s.backward_run(t(lam), s.run(steps, kt), kt)
    s.close()
    for got, want in ((g[0].cpu().numpy(), ref["sigma0"]), (g[1].cpu().numpy(), ref["kappa"]),
                      (np.array(g[2]), np.array(ref["Wi"])), (np.array(g[3]), np.array(ref["beta"]))):
        assert np.max(np.abs(got - want)) < 1e-9 * np.max(np.abs(want))
