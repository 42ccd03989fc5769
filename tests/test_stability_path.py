"""The explicit transport's limit against the search that defines it, every point of it
tested (doubling, then bisection, on polygons whose angles NumPy sums): tables for which
polygons pass the origin at rounding distance and are unstable by a rounding
error far below the limit, which a search that tests fewer points stops at; and
the paper's variable with one exponent, f = delta (1 + c t s zeta (2 - zeta)) up to
1/(mu dt), which vanishes at zeta = 1 whatever t, so that no velocity is let through.

dt 1e-3 to 0.1, one exponent mu = r / dt of weight w r.  The limit is bisected to 1e-7: 3e-7 for two
searches over the same points."""
import math

import numpy as np
import pytest

from test_stability_search import limit


def searched(dt, tab, stencil, form):
    fine = 2 * math.pi / 2048
    tail = fine * 1e-6 ** (np.arange(200, 0, -1) / 200)
    phi = np.concatenate([tail, fine * np.arange(1, 2048), 2 * math.pi - tail[::-1]])
    z = np.exp(1j * phi)
    delta = 1.5 - 2 * z + 0.5 * z * z
    mu, w = tab
    V = (w / (delta[:, None] + mu * dt)).sum(1) * delta
    W, G = (delta, z * (2 - z) * V) if form else (V * dt, z * (2 - z))
    th = 2 * math.pi * np.arange(1, 240) / 240
    s = 1j * np.sin(th) if stencil else (np.exp(-2j * th) - 6 * np.exp(-1j * th) + 3 + 2 * np.exp(1j * th)) / 6

    def stable(t):
        f = W + t * s[:, None] * G
        turn = np.angle(f / np.roll(f, 1, axis=1)).sum(1)
        return not np.any(np.abs(turn) > math.pi)

    lo, hi = 1e-12, 1e-6
    if not stable(lo):
        return 0.0
    while stable(hi) and hi < 1e6:
        lo, hi = hi, 2 * hi
    while hi - lo > 1e-7 * hi:
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if stable(mid) else (lo, mid)
    return lo


@pytest.mark.parametrize("dt,r,w,stencil,form", [(1e-3, 10.0, 30.0, 1, 0), (1e-3, 1e5, 1.0, 1, 0), (1e-2, 1e3, 30.0, 1, 0),
                                                 (0.1, 10.0, 1.0, 1, 0), (1e-2, 10.0, 30.0, 0, 0),
                                                 (1e-3, 1e3, 1.0, 0, 1), (1e-2, 1e5, 30.0, 0, 1), (1e-2, 1e3, 1.0, 1, 1)])
def test_limit_of_the_full_search(dt, r, w, stencil, form):
    tab = (np.array([r / dt]), np.array([w * r]))
    ref = searched(dt, tab, stencil, form)
    got = limit(0.5, dt, 1, tab, stencil, form)
    assert abs(got - ref) <= 3e-7 * ref + 1e-290
    assert (ref == 0.0) == bool(form)
