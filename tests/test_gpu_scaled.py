"""Scaled rotations of the fused kernels (|theta| <= 0.075): the lanes and rows
at the edges of the grid take coefficients of their own, by how the side ends in
a lane's four columns (sides 8 .. 13 and 32 .. 41, around a strip of 112 or 120 columns) and
by its parity, at every depth; the largest angle of the form and the first one
beyond it, which takes the lifting form, as sides 1 .. 7 do at every angle.

Tolerances.  A step rounds each component about 10 times (six sweeps, the phase
and the scale) by at most 2^-24 relative, and 13 steps add up like a random
walk: 2^-24 sqrt(130) = 7e-7, with a factor 3 for the tails and the rounding of
the coefficients: 2e-6.  The scale's rounding adds at most 1e-9 to the norm per
step, the random roundings 2^-24 sqrt(130 / sites), so 13 steps stay within
1.3e-8 + 3 * 7e-7 / sqrt(sites); the input's rounding to FP32 adds up to 2^-23."""
import numpy as np
import pytest

import oracle
from paper_1208_2407_gb300 import trotter
from gpu_helpers import random_state, rel_l2, run_gpu

pytestmark = pytest.mark.gpu

STEPS, TOL = 13, 2e-6
SIDES = [(32, 41), (33, 40), (34, 39), (35, 38), (36, 37), (37, 8), (8, 33), (9, 32), (10, 9),
         (11, 8), (12, 11), (13, 10), (124, 15), (126, 14), (127, 9), (128, 13), (129, 8),
         (240, 10), (241, 9), (114, 9), (115, 10), (120, 11), (121, 12),
         (124, 5), (125, 6), (126, 4), (128, 3), (1, 9), (2, 8), (3, 7), (4, 6), (5, 5), (6, 4),
         (7, 3), (8, 2), (9, 1), (111, 12),
         (112, 13), (113, 14), (114, 5), (115, 6), (116, 33), (119, 8), (120, 7), (121, 6),
         (225, 40), (226, 41)]


@pytest.mark.parametrize("nx,ny", SIDES)
@pytest.mark.parametrize("theta", [0.075, -0.075, 0.0751])
def test_edges_at_every_depth(nx, ny, theta):
    rng = np.random.default_rng(nx * 1009 + ny)
    re, im = random_state(rng, nx, ny)
    V = rng.uniform(-0.5, 0.5, (ny, nx))
    dt = 2.0 * theta
    ore, oim = oracle.evolve(re, im, V, dt, theta, STEPS)
    for K in range(0, 9):
        (gre, gim), _ = run_gpu(re, im, V, dt, theta, STEPS, K=K)
        assert rel_l2(gre, gim, ore, oim) < TOL, K
        drift = abs(np.sum(gre * gre + gim * gim) - np.sum(ore * ore + oim * oim))
        assert drift < 1.3e-8 + 3 * 7e-7 / np.sqrt(nx * ny) + 1.2e-7, (K, drift)


@pytest.mark.parametrize("nx,ny,nz", [(1, 1, 2), (2, 3, 4), (3, 2, 5), (113, 4, 3), (5, 7, 22),
                                      (9, 6, 23)])
@pytest.mark.parametrize("theta", [0.075, 0.0751])
def test_edges_3d(nx, ny, nz, theta):
    rng = np.random.default_rng(nx + 31 * ny + 97 * nz)
    re, im = rng.standard_normal((2, nz, ny, nx))
    s = np.sqrt(np.sum(re * re + im * im))
    re, im = re / s, im / s
    V = rng.uniform(-0.5, 0.5, (nz, ny, nx))
    g = trotter.Grid(nx, ny, "f32", nz=nz)
    try:
        g.set_state(re, im)
        g.set_potential(V, 2.0 * theta, theta)
        g.evolve(STEPS)
        gre, gim = g.get_state(np.float64)
    finally:
        g.close()
    ore, oim = oracle.evolve3(re, im, V, 2.0 * theta, theta, STEPS)
    assert rel_l2(gre, gim, ore, oim) < TOL


def test_batch_of_both_forms_equals_solo_runs():
    """A batch of grids on either side of the largest scaled angle: each form
    has its own launches, and each grid's result is its solo result."""
    rng = np.random.default_rng(5)
    cases = [(130, 66, 0.075, 9), (64, 40, 0.2, 11), (33, 57, 0.0751, 6), (250, 9, 0.01, 7)]
    grids, want = [], []
    try:
        for nx, ny, theta, steps in cases:
            re, im = random_state(rng, nx, ny)
            V = rng.uniform(-0.5, 0.5, (ny, nx))
            g = trotter.Grid(nx, ny, "f32")
            g.set_state(re, im)
            g.set_potential(V, 0.05, theta)
            grids.append(g)
            want.append(run_gpu(re, im, V, 0.05, theta, steps, K=0)[0])
        trotter.evolve_batched(grids, [c[3] for c in cases])
        for g, (wre, wim) in zip(grids, want):
            gre, gim = g.get_state(np.float64)
            assert np.array_equal(gre, wre) and np.array_equal(gim, wim)
    finally:
        for g in grids:
            g.close()


@pytest.mark.parametrize("nx,ny,depth", [(1448, 1448, 3), (1449, 1448, 4)])
def test_default_depth_of_the_lifting_form(nx, ny, depth):
    """Around 2^21 sites, alone and batched: bit for bit the launches of `depth`."""
    rng = np.random.default_rng(nx)
    re, im = random_state(rng, nx, ny)
    V = rng.uniform(-0.5, 0.5, (ny, nx))
    out = []
    for run in (lambda g: g.evolve(13), lambda g: g.evolve(13, depth),
                lambda g: trotter.evolve_batched([g], [13])):
        g = trotter.Grid(nx, ny, "f32")
        try:
            g.set_state(re, im)
            g.set_potential(V, 0.2, 0.1)
            run(g)
            out.append(g.get_state(np.float32))
        finally:
            g.close()
    for r, i in out[1:]:
        assert np.array_equal(r, out[0][0]) and np.array_equal(i, out[0][1])


@pytest.mark.parametrize("nx,ny,K,theta", [(2000, 1, 0, 0.0731), (1, 2000, 0, 0.0731),
                                           (2000, 2, 3, 0.075), (2, 2000, 3, 0.075),
                                           (2000, 4, 0, 0.0731)])
def test_norm_on_grids_that_are_mostly_edge(nx, ny, K, theta):
    """Sides of less than 8 sites take the lifting form, whose steps leave the norm
    alone: what is left is the phase table's rounding, at most 2 s^2 2^-25 = 3.4e-10
    per step and site with s = sin(0.075), of either sign, and the random roundings,
    2^-24 sqrt(10 / (steps sites)) = 7e-11 per step: below 6e-10 together."""
    steps = 4000
    rng = np.random.default_rng(nx)
    re, im = random_state(rng, nx, ny)
    V = rng.uniform(-0.5, 0.5, (ny, nx))
    g = trotter.Grid(nx, ny, "f32")
    try:
        g.set_state(re, im)
        g.set_potential(V, 2.0 * theta, theta)
        before = g.norm()
        g.evolve(steps, K)
        drift = (g.norm() / before - 1.0) / steps
    finally:
        g.close()
    assert abs(drift) < 6e-10, drift
