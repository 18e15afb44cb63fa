"""A row's padding (columns nx up to the pitch) holds anything: a grid's slab may
be memory that another owner has used, and the library writes no table entry past
column nx - 1.  With NaN in the padding of every plane, evolution alone and
batched, the gradient, the fourth-order step and served requests give bit for bit
what they give with zeros there, at sides of every remainder by the four columns
of a lane, on grids that tiles and grids that warp streams run."""
import numpy as np
import pytest

from paper_1208_2407_gb300 import trotter
from gpu_helpers import ensure_library, random_state

pytestmark = pytest.mark.gpu

SIDES = [(301, 130), (242, 65), (983, 48), (3, 9), (129, 40)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_library()


def _poison(g):
    """NaN in the padding of the grid's seven planes."""
    import torch
    L = g.layout
    for i in range(7):
        start = i * int(L.plane_bytes)
        plane = g.slab[start:start + int(L.pitch) * g.ny * 4].view(torch.float32)
        plane.reshape(g.ny, int(L.pitch))[:, g.nx:] = float("nan")
    torch.cuda.synchronize()


def _both(nx, ny, run, theta=0.03, **potential):
    """run(grid) with zeros and with NaN in the padding."""
    rng = np.random.default_rng(nx * 7 + ny)
    re, im = random_state(rng, nx, ny)
    V = rng.uniform(-0.5, 0.5, (ny, nx))
    out = []
    for poison in (False, True):
        g = trotter.Grid(nx, ny, "f32")
        try:
            g.set_state(re, im)
            g.set_potential(V, 0.05, theta, **potential)
            if poison:
                _poison(g)
            out.append(run(g))
        finally:
            g.close()
    for clean, dirty in zip(*out):
        assert np.isfinite(clean).all()
        assert np.array_equal(clean, dirty)


@pytest.mark.parametrize("nx,ny", SIDES + [(1001, 800)])
@pytest.mark.parametrize("theta", [0.03, 0.2])
def test_evolve(nx, ny, theta):
    def run(g):
        for K in (1, 2, 3, 4):
            g.evolve(2 * K + 1, K)
        return g.get_state(np.float64)

    _both(nx, ny, run, theta)


@pytest.mark.parametrize("nx,ny", SIDES)
def test_evolve_batched(nx, ny):
    def run(g):
        other = trotter.Grid(64, 40, "f32")     # (a grid by itself runs as if alone)
        other.set_potential(None, 0.05, 0.03)
        try:
            trotter.evolve_batched([g, other], [11, 11])
            return g.get_state(np.float64)
        finally:
            other.close()

    _both(nx, ny, run)


@pytest.mark.parametrize("nx,ny", SIDES)
def test_gradient(nx, ny):
    rng = np.random.default_rng(1)
    target = random_state(rng, nx, ny)

    def run(g):
        F, grad = trotter.adjoint_fidelity_grad(g, *target, 13, 5)
        return np.float64(F), grad.cpu().numpy()

    _both(nx, ny, run)


@pytest.mark.parametrize("nx,ny", SIDES)
def test_fourth_order_with_its_own_table(nx, ny):
    """The table of the backward substep lies in an allocation of its own, here
    one that likely held NaN before."""
    import torch

    def run(g):
        g.evolve(3, 2)
        return g.get_state(np.float64)

    for _ in range(8):
        junk = torch.full((1 << 19,), float("nan"), device="cuda")
        del junk
        torch.cuda.empty_cache()
    _both(nx, ny, run, 0.1, order=4)


def _nan_words(shape):
    """Finite doubles around 1e-3 whose low words are NaN patterns."""
    bits = np.random.default_rng(2).uniform(1e-3, 2e-3, shape).view(np.uint64)
    return ((bits & np.uint64(0xFFFFFFFF00000000)) | np.uint64(0x7FC00000)).view(np.float64)


@pytest.mark.parametrize("nx,ny", [(301, 400), (402, 300), (303, 390)])
def test_served_request_in_a_used_slab(nx, ny):
    """The server reuses the slabs of released requests as they are.  A 512 x 512
    request without steps leaves its FP64 inputs in the idle planes, where the
    next request's smaller slab has its tables."""
    junk = _nan_words((512, 512))
    rng = np.random.default_rng(nx)
    re, im = random_state(rng, nx, ny)
    V = rng.uniform(-0.5, 0.5, (ny, nx))
    srv = trotter.Server(hbm_budget_bytes=1 << 30, max_slots=1)
    try:
        t = srv.submit(512, 512, 0, 0.05, 0.03, junk, junk, junk)
        assert srv.wait(t, 60000).status == 0
        srv.release(t)
        t = srv.submit(nx, ny, 9, 0.05, 0.03, V, re, im)
        assert srv.wait(t, 60000).status == 0
        got = srv.fetch(t, ny, nx)
        srv.release(t)
    finally:
        srv.close()
    g = trotter.Grid(nx, ny, "f32")
    try:
        g.set_state(re, im)
        g.set_potential(V, 0.05, 0.03)
        g.evolve(9, 4)
        want = g.get_state(np.float64)
    finally:
        g.close()
    assert np.isfinite(want[0]).all()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
