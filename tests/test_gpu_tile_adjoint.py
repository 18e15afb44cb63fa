"""The backward adjoint on tiles: sides that put the grid's edges and the last
tile at every place of a tile (48 rows, 36 or 32 of them stored, strips of 112
columns, sides of 1 to 9), angles of either kind (|theta| > 0.075 takes the
lifting streams), depths 2 to 4 and the default, against the FP64 oracle
adjoint.  Tolerance: the FP32 states err by 2^-24 sqrt(10 n) after n steps (see
test_gpu_scaled.py), forward and backward and in both factors of a term, 4 times
that in all: 5e-6 for 14 steps, with a factor 4 for small grids: 2e-5."""
import numpy as np
import pytest

import oracle
from gpu_helpers import random_state
from test_gpu_adjoint import gpu_adjoint, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(1, 3), (2, 9), (3, 48), (4, 49), (9, 47), (112, 80), (113, 81),
                                   (128, 84), (129, 33), (241, 130)])
@pytest.mark.parametrize("theta", [0.025, 0.075, 0.0751])
def test_gradient(nx, ny, theta):
    rng = np.random.default_rng(nx * 7 + ny)
    re, im = random_state(rng, nx, ny)
    tre, tim = random_state(rng, nx, ny)
    tre, tim = 0.6 * re + 0.4 * tre, 0.6 * im + 0.4 * tim   # so that F is not tiny
    s = np.sqrt(np.sum(tre ** 2 + tim ** 2))
    tre, tim = tre / s, tim / s
    V = rng.uniform(-0.5, 0.5, (ny, nx))
    c = dict(nx=nx, ny=ny, re=re, im=im, target_re=tre, target_im=tim, V=V, dt=2 * theta,
             theta=theta)
    og, oF, _ = oracle.adjoint_grad(re, im, tre, tim, V, 2 * theta, theta, 14)
    for K in (0, 2, 3, 4):
        F, g = gpu_adjoint(c, 14, 9, K)   # segments of 9 and 5 steps: remainders of 1 to 3
        assert rel(g, og) < 2e-5, (K, rel(g, og))
