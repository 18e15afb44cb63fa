"""Read-backs of many grids: results land in pinned slots that calls hold while they
wait, so grids come and go without pinned memory being made or freed (freeing it
waits for the device), and more readers at a time than there are slots still read
their own results."""
import threading

import pytest

from paper_1208_2407_gb300 import trotter
from gpu_helpers import ensure_library

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_library()


def _grid(i, stream=None):
    """A grid whose norm is 64 * 32 * i * i."""
    import torch
    g = trotter.Grid(64, 32, "f32")
    v = torch.full((32, 64), float(i), device="cuda")
    g.set_state(v, torch.zeros_like(v), stream)
    torch.cuda.synchronize()
    return g


def test_closing_many_grids_does_not_wait_for_the_device():
    import torch
    grids = [_grid(i) for i in range(130)]
    for i, g in enumerate(grids):
        assert g.norm() == 64 * 32 * i * i
    big = trotter.Grid(8192, 8192, "f32")
    try:
        big.set_potential(None, 0.05, 0.025)
        stream, done = torch.cuda.Stream(), torch.cuda.Event()
        with torch.cuda.stream(stream):
            big.evolve(6000)              # about 0.4 s
            done.record()
        for g in grids:
            g.close()
        assert not done.query()
        torch.cuda.synchronize()
    finally:
        big.close()


def test_more_readers_than_slots():
    import torch
    n = 80
    grids = [_grid(i) for i in range(n)]
    ready = threading.Barrier(n)
    bad = []

    def read(i):
        st = torch.cuda.Stream()
        ready.wait()
        for _ in range(20):
            v = grids[i].norm(trotter._VP(st.cuda_stream))
            if v != 64 * 32 * i * i:
                bad.append((i, v))

    threads = [threading.Thread(target=read, args=(i,)) for i in range(n)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for g in grids:
        g.close()
    assert not bad
