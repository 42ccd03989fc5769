"""The transposed transport stencil: one reverse step with kappa = 0, where the adjoint of the right-hand side is
known from the gradient without transport; the sum of its 13 (2D 9) FP64
products within 30 rounding errors of the sum of their magnitudes. In FP32
storage too the sum is one of FP64 products, also where the values are so small (dJ
scaled by 2^-100) that a float product's rounding error is no longer representable, or
so large (2^112) that the scaled weights' products leave the float range."""
import numpy as np
import pytest

from helpers import ensure_lib
from test_gpu_run import problem, solver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def transposed(case, u, lam):
    """A^T lam and |A|^T |lam| of A = dt (u.grad_h - eps Lap_h), numpy FP64."""
    n, dim = case["n"], case["dim"]
    out, mag = np.zeros_like(lam), np.zeros_like(lam)
    for a in range(dim):
        h = 2 * np.pi / n[a]
        up = u[a] >= 0.0
        taps = {-1: -3.0 + 0 * u[a], 1: 3.0 + 0 * u[a]} if case["stencil"] else \
            {-2: np.where(up, 1.0, 0.0), -1: np.where(up, -6.0, -2.0), 0: np.where(up, 3.0, -3.0),
             1: np.where(up, 2.0, 6.0), 2: np.where(up, 0.0, -1.0)}
        for k in range(-2, 3):
            c = case["dt"] * u[a] * taps.get(k, 0.0) / (6 * h)
            c = c - case["eps"] * case["dt"] / h ** 2 * {0: -2.0, 1: 1.0, -1: 1.0}.get(k, 0.0)
            axis = dim - 1 - a           # x fastest
            term = (c * lam).reshape((-1,) + n[::-1])
            term = np.roll(term, k, axis=1 + axis).reshape(lam.shape)
            out += term
            mag += np.abs(term)
    return out, mag


@pytest.mark.parametrize("dim,n,stencil,eps", [(2, (37, 5), 0, 0.0), (2, (8, 8), 1, 1e-3), (2, (5, 3), 0, 1e-3),
                                               (3, (9, 5, 4), 0, 1e-3), (3, (6, 1, 7), 0, 0.0), (3, (8, 4, 4), 1, 0.0)])
@pytest.mark.parametrize("exponent", [0, -100, 112])
@pytest.mark.parametrize("precision", [0, 1])
def test_transposed_stencil(dim, n, stencil, eps, exponent, precision):
    import torch
    case, kap, u, sigma0, lam = problem(dim, n, 5, 1, True, stencil, eps)
    grads = []
    for moving in (False, True):
        s = solver(dict(case, transport=moving, eps=case["eps"] if moving else 0.0), precision)
        t = lambda a: torch.as_tensor(a, dtype=s.dtype, device="cuda").contiguous()
        kt, ut = t(0.0 * kap), t(u) if moving else None
        s.set_state(t(sigma0))
        grads.append(s.backward_run(t(np.ldexp(lam, exponent)), s.run(1, kt, ut), kt, ut)[0].cpu().numpy())
        s.close()
    mu, w, dt = case["mu"], case["w"], case["dt"]
    eta = float(np.sum(1.5 * w * dt / (1.5 + mu * dt)))
    lamR = grads[0] / eta                          # dJ/dsigma0 = eta lamR without transport
    if precision == 1:
        lamR = lamR.astype(np.float32).astype(np.float64)
    # E = 2 sigma^0 - sigma^{-1} = sigma0: dJ/dsigma0 gains -A^T lamR
    At, mag = transposed(case, u, lamR)
    err = np.abs(grads[1] - (grads[0] - At))
    eps64 = 1.2e-16
    # besides the sum: lamE enters as 2 lamE - lamE, lamR is known to two roundings, eta lamR to one
    assert np.all(err <= eps64 * (30 * mag + 8 * np.abs(grads[0]) + 1e-30 * mag.max()))
