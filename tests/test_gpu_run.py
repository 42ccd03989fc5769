"""Runs with a frozen velocity gradient in one call (tfs_run, tfs_backward_run, and
tfs_backward on the same kernels) at the sizes where they can go wrong: tiles
that end past the grid, numbers of modes around the unrolled groups of eight and
the register variants, the largest table, more steps than one launch takes, no
initial stress, both stencils with and without diffusion.  Against the FP64
oracle at the bounds the single steps are held to (2e-5 normwise for the FP32
stress, 2e-4 for the FP32 gradients, 1e-11 and 1e-10 in FP64), and bitwise against
stepping."""
import numpy as np
import pytest

from helpers import ensure_lib, rel_err_per_component, stable_velocity
from oracle import orc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def problem(dim, n, m, steps, transport, stencil=0, eps=0.0, alpha=0.5, dt=2e-3, seed=11):
    mu = np.geomspace(0.1, 2.0 / dt, m) if m > 1 else np.array([3.0])
    h = np.log(mu[1] / mu[0]) if m > 1 else 1.0
    w = h * np.sin(np.pi * alpha) / np.pi * mu ** alpha
    rng = np.random.default_rng(seed)
    N, nc = int(np.prod(n)), 3 if dim == 2 else 6
    f32 = lambda a: np.asarray(a, np.float32).astype(np.float64)
    case = dict(dim=dim, n=n, alpha=alpha, Wi=1.3, beta=0.4, dt=dt, mu=mu, w=w, stencil=stencil,
                eps=eps if transport else 0.0, transport=transport)
    u = rng.normal(size=(dim, N))
    if transport:
        u = stable_velocity(case, u, 0.5)
    # inputs representable in float, so that both storage forms and the oracle take the same ones
    return case, f32(0.3 * rng.normal(size=(dim * dim, N))), f32(u), f32(0.3 * rng.normal(size=(nc, N))), \
        f32(rng.normal(size=(nc, N)))


def oracle_problem(case):
    return orc.Problem(**{k: case[k] for k in ("dim", "n", "alpha", "Wi", "beta", "dt", "mu", "w", "eps", "stencil",
                                               "transport")})


def solver(case, precision):
    from paper_2411_17294_gb300 import tfs
    return tfs.Solver(case["dim"], case["n"], case["alpha"], case["Wi"], case["beta"], case["dt"], m=len(case["mu"]),
                      precision=precision, mu=case["mu"], w=case["w"], transport=case["transport"], eps=case["eps"],
                      stencil=case["stencil"])


CASES = [(2, (5, 3), 1, 1, False, 0, 0.0), (2, (43, 3), 8, 7, False, 0, 0.0), (2, (9, 5), 17, 131, False, 0, 0.0),
         (3, (5, 5, 3), 48, 4, False, 0, 0.0), (2, (8, 4), 64, 5, False, 0, 0.0), (3, (4, 3, 2), 55, 6, False, 0, 0.0), (2, (32, 4), 9, 8, True, 0, 0.0),
         (2, (13, 10), 64, 9, True, 1, 1e-4), (2, (1, 1), 4, 17, False, 0, 0.0), (2, (7, 2), 5, 2, True, 0, 1e-4),
         (3, (5, 4, 7), 6, 16, False, 0, 0.0), (3, (6, 5, 4), 3, 10, True, 0, 0.0), (3, (8, 4, 4), 33, 11, True, 1, 1e-4),
         (3, (3, 2, 1), 2, 3, True, 0, 1e-3)]


@pytest.mark.parametrize("dim,n,m,steps,transport,stencil,eps", CASES)
@pytest.mark.parametrize("zero", [False, True])
def test_run_matches_oracle_and_leaves_the_state(dim, n, m, steps, transport, stencil, eps, zero):
    import torch
    case, kap, u, sigma0, _ = problem(dim, n, m, steps, transport, stencil, eps)
    o = orc.Oracle(oracle_problem(case), None if zero else sigma0)
    ref = []
    for _ in range(steps + 3):
        o.step(kap, kap, u)
        ref.append(o.sig_n.copy())
    for precision, tol in ((1, 2e-5), (0, 1e-11)):
        s = solver(case, precision)
        t = lambda a: torch.as_tensor(a, dtype=s.dtype, device="cuda").contiguous()
        kt, ut = t(kap), t(u)
        s.set_state(None if zero else t(sigma0))
        got = s.run(steps, kt, ut if transport else None)
        assert s.step_index() == steps
        assert torch.equal(s.stress(), got[-1])
        for _ in range(3):
            s.step(kt, kt, ut if transport else None)
        assert np.all(rel_err_per_component(s.stress().double().cpu().numpy(), ref[-1]) < tol)
        got = got.double().cpu().numpy()
        for k in range(steps):
            assert np.all(rel_err_per_component(got[k], ref[k]) < tol), (precision, k)
        assert s.status() == 0
        s.close()


@pytest.mark.parametrize("dim,n,m,steps,transport,stencil,eps", CASES)
@pytest.mark.parametrize("K", [0, 3, 8])
def test_reverse_matches_oracle(dim, n, m, steps, transport, stencil, eps, K):
    # K = 0: from the trajectory; else from checkpoints every K steps
    import torch
    case, kap, u, sigma0, lam = problem(dim, n, m, steps, transport, stencil, eps)
    ref = orc.gradients(oracle_problem(case), sigma0, kap, u, steps, lam)
    for precision, tol in ((1, 2e-4), (0, 1e-10)):
        s = solver(case, precision)
        t = lambda a: torch.as_tensor(a, dtype=s.dtype, device="cuda").contiguous()
        kt, ut = t(kap), t(u) if transport else None
        s.set_state(t(sigma0))
        if K == 0:
            g = s.backward_run(t(lam), s.run(steps, kt, ut), kt, ut)
        else:
            ckpts = []
            for k in range(steps):
                if k % K == 0:
                    ckpts.append(s.new_checkpoint())
                    s.save(ckpts[-1])
                s.step(kt, kt, ut)
            g = s.backward(t(lam), ckpts, K, steps, kt, ut)
        s.close()
        for got, want in ((g[0].cpu().numpy(), ref["sigma0"]), (g[1].cpu().numpy(), ref["kappa"]),
                          (np.array([[g[2]]]), np.array([[ref["Wi"]]])), (np.array([[g[3]]]), np.array([[ref["beta"]]]))):
            assert np.max(np.abs(got - want)) < tol * np.max(np.abs(want)), precision


@pytest.mark.parametrize("dim,n,m,steps,transport,stencil,eps", CASES)
@pytest.mark.parametrize("precision", [0, 1, 2])
def test_run_is_stepping_bitwise(dim, n, m, steps, transport, stencil, eps, precision):
    import torch
    case, kap, u, sigma0, _ = problem(dim, n, m, steps, transport, stencil, eps)
    a, b = solver(case, precision), solver(case, precision)
    t = lambda v: torch.as_tensor(v, dtype=a.dtype, device="cuda").contiguous()
    kt, ut = t(kap), t(u) if transport else None
    a.set_state(t(sigma0))
    b.set_state(t(sigma0))
    rows = a.run(steps, kt, ut)
    for k in range(steps):
        b.step(kt, kt, ut)
        assert torch.equal(rows[k], b.stress()), k
    ca, cb = a.new_checkpoint().zero_(), b.new_checkpoint().zero_()   # modes and stress levels too
    a.save(ca)
    b.save(cb)
    assert torch.equal(ca[256:], cb[256:])
    a.close()
    b.close()


def test_refusals():
    import torch
    from paper_2411_17294_gb300 import tfs
    case, kap, u, sigma0, lam = problem(2, (8, 4), 4, 3, False)
    s = solver(case, 1)
    t = lambda a: torch.as_tensor(a, dtype=s.dtype, device="cuda").contiguous()
    kt = t(kap)
    with pytest.raises(tfs.TfsError) as err:      # no state
        s.run(3, kt)
    assert err.value.code == tfs.TFS_ERR_STATE
    s.set_state(t(sigma0))
    with pytest.raises(tfs.TfsError) as err:
        s.run(0, kt)
    assert err.value.code == tfs.TFS_ERR_ARG
    s.close()
    m = tfs.Solver(2, (8, 4), 0.5, 1.0, 0.5, 1e-3, m=4, precision=1, mu=case["mu"], w=case["w"], transport=True)
    m.set_state(t(sigma0))
    with pytest.raises(tfs.TfsError) as err:      # transport without a velocity
        m.run(2, kt)
    assert err.value.code == tfs.TFS_ERR_ARG
    m.close()
