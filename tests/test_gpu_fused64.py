"""Fused FP64 steps (one launch per step) against the oracle: sides around the
strips of 26, 58 and 122 columns and the row ranges, odd and even, sides of one
to three, positive, negative and largest angles, the fourth-order step, and a
run long enough to be cut where the scaled state has grown by 2^30.

Tolerance: about 20 roundings of 2^-53 per component and step that add up like a
random walk, and coefficients within 2^-53 that add up linearly over the steps:
n steps stay within 2^-53 (3 sqrt(20 n) + 10 n), below 1e-13 for 20 steps and
2e-12 for 1500."""
import numpy as np
import pytest

import oracle
from paper_1208_2407_gb300 import trotter
from gpu_helpers import random_state, rel_l2, run_gpu

pytestmark = pytest.mark.gpu

SIDES = [(1, 1024), (1024, 1), (2, 600), (600, 2), (3, 401), (401, 3), (25, 57), (26, 58),
         (27, 59), (57, 40), (58, 33), (121, 30), (122, 31), (123, 64), (250, 123), (513, 37)]


@pytest.mark.parametrize("nx,ny", SIDES)
@pytest.mark.parametrize("theta", [0.025, -0.1, 0.39])
def test_matches_oracle(nx, ny, theta):
    rng = np.random.default_rng(nx * 31 + ny)
    re, im = random_state(rng, nx, ny)
    V = rng.uniform(-0.5, 0.5, (ny, nx))
    for steps in (1, 2, 9):
        (gre, gim), _ = run_gpu(re, im, V, 2.0 * theta, theta, steps, dtype="f64")
        ore, oim = oracle.evolve(re, im, V, 2.0 * theta, theta, steps)
        assert rel_l2(gre, gim, ore, oim) < 1e-13, steps


@pytest.mark.parametrize("nx,ny", [(64, 33), (151, 60)])
def test_order4(nx, ny):
    rng = np.random.default_rng(nx)
    re, im = random_state(rng, nx, ny)
    V = rng.uniform(-0.5, 0.5, (ny, nx))
    g = trotter.Grid(nx, ny, "f64")
    try:
        g.set_state(re, im)
        g.set_potential(V, 0.1, 0.05, order=4)
        planes = g.state_planes()
        trotter.ts_launch_count(reset=True)
        g.evolve(3)
        assert trotter.ts_launch_count() == 5 * 3 + 3    # 2 sweeps, a launch per substep, the tail
        assert g.state_planes() == planes                # the state stays in its planes
        gre, gim = g.get_state(np.float64)
    finally:
        g.close()
    ore, oim = oracle.evolve(re, im, V, 0.1, 0.05, 3, order=4)
    assert rel_l2(gre, gim, ore, oim) < 1e-13


def test_long_run_is_cut():
    # theta = 0.39: a step grows the bulk by 1.64 per axis (two odd sweeps at theta and
    # an even one at 2 theta), 2.7 in all, so 2^30 is passed every 21 steps
    rng = np.random.default_rng(2)
    re, im = random_state(rng, 45, 34)
    V = rng.uniform(-0.5, 0.5, (34, 45))
    (gre, gim), _ = run_gpu(re, im, V, 0.78, 0.39, 1500, dtype="f64")
    ore, oim = oracle.evolve(re, im, V, 0.78, 0.39, 1500)
    assert rel_l2(gre, gim, ore, oim) < 2e-12
