"""Tiles held in registers against the warp streams: which of the two runs a
launch is a matter of speed alone, so an evolution whose launches are tiles
must give bit for bit what the streams give.  A driven grid with V1 = 0 runs the
streams (a drive phase of zero angle leaves every bit), so it is the reference
here; sides put the grid's edges and its last tile at every place of a tile
(sides of 8 to 13, around 112 columns and 16, 24 and 48 rows, ragged; smaller sides
take the lifting form, streams in both runs)."""
import numpy as np
import pytest

import oracle
from paper_1208_2407_gb300 import trotter
from gpu_helpers import random_state, rel_l2

pytestmark = pytest.mark.gpu

SIDES = [(8, 8), (9, 11), (10, 24), (11, 25), (12, 9), (13, 47), (128, 30), (240, 32), (241, 65),
         (1, 1), (2, 5), (3, 9), (4, 17), (5, 24), (9, 25), (111, 48), (112, 49), (113, 16),
         (225, 33), (300, 47), (130, 97), (7, 200), (500, 301)]


@pytest.mark.parametrize("nx,ny", SIDES)
@pytest.mark.parametrize("K", [1, 2, 3, 4])
def test_tiles_equal_streams(nx, ny, K):
    rng = np.random.default_rng(nx * 1009 + ny + K)
    re, im = random_state(rng, nx, ny)
    V = rng.uniform(-0.5, 0.5, (ny, nx))
    steps = 2 * K + 1                       # launches of depth K and one of depth 1
    out = []
    for drive in (False, True):
        g = trotter.Grid(nx, ny, "f32")
        try:
            g.set_state(re, im)
            g.set_potential(V, 0.05, 0.03)
            if drive:
                g.set_drive(None, np.ones(steps))
            g.evolve(steps, K)
            out.append(g.get_state(np.float64))
        finally:
            g.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    ore, oim = oracle.evolve(re, im, V, 0.05, 0.03, steps)
    assert rel_l2(*out[0], ore, oim) < 2e-6     # as derived in test_gpu_scaled.py


# grids that tiles of 80 rows cover in one round of one block per SM where tiles
# of 64 rows take two: the fewest and the most rows of that range, ragged sides
@pytest.mark.parametrize("nx,ny", [(1024, 785), (1023, 1039), (1017, 1040), (897, 911)])
@pytest.mark.parametrize("K", [3, 4])
def test_tall_tiles_equal_streams(nx, ny, K):
    test_tiles_equal_streams(nx, ny, K)


def test_captured_evolution():
    """Dependent launches inside a CUDA graph keep their order: three replays
    of a captured evolution equal three evolutions."""
    import torch
    rng = np.random.default_rng(3)
    re, im = random_state(rng, 200, 90)
    V = rng.uniform(-0.5, 0.5, (90, 200))
    outs = []
    for captured in (False, True):
        g = trotter.Grid(200, 90, "f32")
        try:
            g.set_state(re, im)
            g.set_potential(V, 0.05, 0.025)
            torch.cuda.synchronize()
            if captured:
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph):
                    g.evolve(32)          # an even number of launches: the planes return
                for _ in range(3):
                    graph.replay()
            else:
                for _ in range(3):
                    g.evolve(32)
            torch.cuda.synchronize()
            outs.append(g.get_state(np.float64))
        finally:
            g.close()
    assert np.array_equal(outs[0][0], outs[1][0]) and np.array_equal(outs[0][1], outs[1][1])


def test_potential_set_under_capture_then_again():
    """A captured set_potential has not run: the next one at the same angle still
    writes what a multi-grid launch reads."""
    import torch

    n, theta = 200, 0.03
    gen = torch.Generator(device="cuda").manual_seed(1)
    V = torch.rand(n, n, dtype=torch.float64, device="cuda", generator=gen)
    re, im = torch.randn(2, n, n, device="cuda", generator=gen)
    grids = [trotter.Grid(n, n, "f32") for _ in range(3)]
    try:
        for g in grids:
            g.set_state(re, im)
        torch.cuda.synchronize()
        with torch.cuda.graph(torch.cuda.CUDAGraph()):
            grids[0].set_potential(V, 2.0 * theta, theta)
        for g in grids:
            g.set_potential(V, 2.0 * theta, theta)
        trotter.evolve_batched([grids[0], grids[2]], [8, 8], 4)   # (one alone is no batch)
        grids[1].evolve(8, 4)
        a, b = (g.get_state(np.float32) for g in grids[:2])
    finally:
        for g in grids:
            g.close()
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
