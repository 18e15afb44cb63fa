"""Observables and norms where the block split of the reduction changes: one
block, a part of a block, one to four blocks per SM, rows of 1 to 5 sites, 3-D.
Against compensated FP64 sums on the host of the same rounded state.  FP32 grids
sum exact products in double-float (48 bits), so a relative error of 1e-13 of
the sum of absolute terms leaves a factor of 30; FP64 grids round every term
(2^-53) and compensate: 1e-14."""
import math

import numpy as np
import pytest

from paper_1208_2407_gb300 import trotter

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (3, 2, 1), (5, 41, 1), (64, 64, 1), (1021, 640, 1), (3001, 1700, 1),
          (7, 5, 3), (130, 66, 40)]


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("nx,ny,nz", SHAPES)
def test_observables(nx, ny, nz, dtype):
    rng = np.random.default_rng(nx + ny)
    shape = (nz, ny, nx) if nz > 1 else (ny, nx)
    t = np.float32 if dtype == "f32" else np.float64
    re, im = (rng.standard_normal(shape).astype(t) for _ in range(2))
    V = rng.uniform(-0.5, 0.5, shape).astype(t).astype(np.float64)
    g = trotter.Grid(nx, ny, dtype, nz=nz)
    try:
        g.set_state(re, im)
        g.set_potential(V, 0.05, 0.025)
        o, n = g.observe(), g.norm()
    finally:
        g.close()
    r, m = re.astype(np.longdouble).reshape(nz, ny, nx), im.astype(np.longdouble).reshape(nz, ny, nx)
    p = r * r + m * m
    tol = 1e-13 if dtype == "f32" else 1e-14
    nrm = p.sum()
    assert abs(o["norm"] - nrm) <= tol * nrm and abs(n - nrm) <= tol * nrm
    c = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    for name, q in (("x", c[2]), ("y", c[1]), ("x2", c[2] ** 2), ("y2", c[1] ** 2)):
        want = (q * p).sum() / nrm
        assert abs(o[name] - want) <= 2 * tol * max(want, 1.0), name
    kin = mag = np.longdouble(0)
    for ax in range(3):
        a = [slice(None)] * 3
        b = [slice(None)] * 3
        a[ax], b[ax] = slice(1, None), slice(None, -1)
        t1 = r[tuple(a)] * r[tuple(b)] + m[tuple(a)] * m[tuple(b)]
        kin, mag = kin + t1.sum(), mag + np.abs(t1).sum()
    assert abs(o["e_kin"] + 2.0 * kin) <= 2 * tol * max(2.0 * mag, 1e-300)
    pot = (V.reshape(p.shape) * p)
    assert abs(o["e_pot"] - pot.sum()) <= tol * np.abs(pot).sum()
    assert math.isfinite(o["z"])
