"""The explicit transport's limit against the definition it searches for: with the
sampled contour of the library's stability test, the polygons W + t s G (angles
summed with NumPy, every direction) wind about the origin just above the limit
and not just below it.  The limit is bisected to 1e-7, so 3e-7 on either side
decides."""
import ctypes
import math

import numpy as np
import pytest

from helpers import ensure_lib
from oracle import soe


def limit(alpha, dt, m, table, stencil, form):
    ensure_lib()
    from paper_2411_17294_gb300 import tfs
    lib = tfs.load_library()
    g = tfs.TfsGrid()
    g.dim = 2
    for a in range(3):
        g.n[a], g.L[a] = (24, 3.0) if a < 2 else (1, 1.0)
    h = ctypes.c_void_p()
    tfs.check(lib.tfs_create(ctypes.byref(h), ctypes.byref(g), alpha, 1.0, 0.5, m, dt, 0), "create")
    tfs.check(lib.tfs_set_param(h, tfs.TFS_PARAM_STENCIL, float(stencil)), "stencil")
    if form:
        tfs.check(lib.tfs_set_param(h, tfs.TFS_PARAM_FORM, 1.0), "form")
    if m:
        mu, w = (np.ascontiguousarray(a, dtype=np.float64) for a in table)
        dp = ctypes.POINTER(ctypes.c_double)
        tfs.check(lib.tfs_set_soe(h, mu.ctypes.data_as(dp), w.ctypes.data_as(dp), m), "soe")
    U = ctypes.c_double(0.0)
    tfs.check(lib.tfs_transport_limit(h, ctypes.byref(U)), "limit")
    lib.tfs_destroy(h)
    return U.value * dt * 2 * (24 / 3.0) / 0.9


def winds(t, alpha, dt, table, stencil, form):
    fine = 2 * math.pi / 2048
    tail = fine * 1e-6 ** (np.arange(200, 0, -1) / 200)
    phi = np.concatenate([tail, fine * np.arange(1, 2048), 2 * math.pi - tail[::-1]])
    z = np.exp(1j * phi)
    delta = 1.5 - 2 * z + 0.5 * z * z
    mu, w = table if table is not None else (np.zeros(0), np.zeros(0))
    V = (w / (delta[:, None] + mu * dt)).sum(1) * delta if len(mu) else None
    W = delta if form or V is None else V * dt
    G = z * (2 - z) * (V if form else 1.0)
    th = 2 * math.pi * np.arange(1, 240) / 240
    s = 1j * np.sin(th) if stencil else (np.exp(-2j * th) - 6 * np.exp(-1j * th) + 3 + 2 * np.exp(1j * th)) / 6
    f = W + t * s[:, None] * G
    turn = np.angle(f / np.roll(f, 1, axis=1)).sum(1)
    return bool(np.any(np.abs(turn) > math.pi))


@pytest.mark.parametrize("alpha,dt,m,stencil,form", [(0.5, 1e-3, 8, 0, 0), (0.5, 1e-3, 8, 1, 0), (0.9, 2e-4, 16, 0, 0),
                                                     (0.3, 5e-3, 4, 1, 0), (1.0, 1e-3, 0, 0, 0), (1.0, 1e-3, 0, 1, 0),
                                                     (0.6, 1e-3, 8, 0, 1), (0.8, 1e-3, 16, 0, 1)])
def test_limit_is_where_the_polygons_start_to_wind(alpha, dt, m, stencil, form):
    table = soe.soe_build(1 - alpha if form else alpha, dt, 50 * dt, m) if m else None
    lam = limit(alpha, dt, m, table, stencil, form)
    assert lam > 0
    assert not winds(lam * (1 - 3e-7), alpha, dt, table, stencil, form)
    assert winds(lam * (1 + 3e-7), alpha, dt, table, stencil, form)
