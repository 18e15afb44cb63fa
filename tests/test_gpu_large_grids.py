"""Grids far larger than L2, where depths 1 to 3 take other kernels and strips than
below (more than 800 MB at 24 bytes per site; driven ones from 4 million sites):
long thin and ragged ones, against depth 4, whose kernel is the same at every size.

Tolerance.  Two runs of 5 steps that round differently: each rounds a component
about 10 times per step by at most 2^-24 relative, which add up like a random walk
to 2^-24 sqrt(50) = 4e-7 of the norm; 2e-6 for two runs with a factor 2 for the
tails and the coefficients' rounding.  The bands at the grid's edges, where a wrong
strip boundary would show, are held to the same."""
import numpy as np
import pytest

from paper_1208_2407_gb300 import trotter

pytestmark = pytest.mark.gpu

TOL = 2e-6
SIDES = [(1003, 33501), (33503, 1001), (5801, 5800), (37, 1000003), (124, 280002),
         (125, 280003)]


def _evolve(nx, ny, theta, K, steps=5, batched=False, drive=False):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(nx)
    g = trotter.Grid(nx, ny, "f32")
    try:
        re, im = (torch.randn((ny, nx), device="cuda", generator=gen) for _ in range(2))
        g.set_state(re, im)
        V = torch.rand((ny, nx), device="cuda", dtype=torch.float64, generator=gen) - 0.5
        g.set_potential(V, 0.05, theta)
        if drive:
            g.set_drive(V, np.linspace(0.5, 1.0, steps))
        if batched:
            other = trotter.Grid(64, 40, "f32")     # (a grid by itself runs as if alone)
            other.set_potential(None, 0.05, theta)
            trotter.evolve_batched([other, g], [steps, steps], K)
            torch.cuda.synchronize()
            other.close()
        else:
            g.evolve(steps, K)
        return torch.stack(g.get_state(np.float32, device=True))
    finally:
        g.close()


def _close(a, b):
    import torch
    bands = [np.s_[:, :, :], np.s_[:, :, :130], np.s_[:, :, -130:], np.s_[:, :9], np.s_[:, -9:]]
    for s in bands:
        x, y = a[s].double(), b[s].double()
        assert float(torch.linalg.norm(x - y) / torch.linalg.norm(y)) < TOL, s


@pytest.mark.parametrize("nx,ny", SIDES)
@pytest.mark.parametrize("theta", [0.05, 0.3])
def test_depths_agree(nx, ny, theta):
    want = _evolve(nx, ny, theta, 4)
    for K in (1, 2, 3):
        _close(_evolve(nx, ny, theta, K), want)


@pytest.mark.parametrize("nx,ny", [(2501, 2400), (301, 20001)])
def test_driven(nx, ny):
    want = _evolve(nx, ny, 0.3, 4, drive=True)
    _close(_evolve(nx, ny, 0.3, 3, drive=True), want)


@pytest.mark.parametrize("K", [2, 4])
def test_batched_equals_alone(K):
    """Depth 2 changes its form with the size, as full launches (K = 2) and as the
    remainder of 6 steps at depth 4, in a batch as alone."""
    import torch
    nx, ny = SIDES[0]
    assert torch.equal(_evolve(nx, ny, 0.05, K, 6), _evolve(nx, ny, 0.05, K, 6, batched=True))
