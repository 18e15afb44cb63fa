"""Batches and servers whose grids take different kernels (scaled rotations, the
lifting form at depth 3, and at depth 4): what runs side by side on a second stream
must see what the caller's stream did before and be seen by what it does after, and
every grid gets bit for bit its solo result, whether its group is one grid or
several, and on either side of the most sites that run side by side."""
import numpy as np
import pytest

from paper_1208_2407_gb300 import trotter
from gpu_helpers import ensure_library

pytestmark = pytest.mark.gpu

# (nx, ny, theta, steps)
MIXES = {
    "one of each": [(200, 90, 0.05, 9), (130, 66, 0.2, 13)],
    "several of each": [(200, 90, 0.05, 9), (64, 64, 0.2, 5), (333, 120, 0.07, 14),
                        (130, 66, 0.3, 13), (512, 512, 0.03, 40)],
    "three kernels": [(300, 300, 0.05, 8), (256, 256, 0.2, 8), (200, 200, 0.2, 11),
                      (1500, 1500, 0.2, 6)],
    "one by one": [(3000, 2400, 0.05, 6), (2100, 2000, 0.2, 6), (64, 64, 0.01, 6)],
}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_library()


def _inputs(nx, ny):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(nx * 31 + ny)
    re, im = (torch.randn((ny, nx), device="cuda", generator=gen) for _ in range(2))
    V = torch.rand((ny, nx), device="cuda", dtype=torch.float64, generator=gen) - 0.5
    return re, im, V


def _grids(mix):
    grids = []
    for nx, ny, theta, _ in mix:
        g = trotter.Grid(nx, ny, "f32")
        g.set_potential(_inputs(nx, ny)[2], 0.05, theta)
        grids.append(g)
    return grids


@pytest.mark.parametrize("name", MIXES)
@pytest.mark.parametrize("own_stream", [False, True])
def test_batch_equals_solo_runs_in_stream_order(name, own_stream):
    import torch
    mix = MIXES[name]
    data = [_inputs(nx, ny) for nx, ny, _, _ in mix]
    steps = [s for *_, s in mix]
    grids = _grids(mix)
    want = []
    try:
        for g, (re, im, _), s in zip(grids, data, steps):
            g.set_state(re, im)
            g.evolve(s)
            want.append(g.get_state(np.float32, device=True))
        torch.cuda.synchronize()
        with torch.cuda.stream(torch.cuda.Stream() if own_stream else torch.cuda.default_stream()):
            for _ in range(5):
                # states set just before, read and overwritten just after
                for g, (re, im, _) in zip(grids, data):
                    g.set_state(re, im)
                trotter.evolve_batched(grids, steps)
                out = [torch.stack(g.get_state(np.float32, device=True)) for g in grids]
                for g, (re, im, _) in zip(grids, data):
                    g.set_state(im, re)
                torch.cuda.current_stream().synchronize()
                for o, w in zip(out, want):
                    assert torch.equal(o, torch.stack(w))
    finally:
        for g in grids:
            g.close()


@pytest.mark.parametrize("name", ["several of each", "one by one"])
def test_server_equals_solo_runs(name):
    mix = [(nx, ny, theta, 3 * s) for nx, ny, theta, s in MIXES[name]]
    data = [_inputs(nx, ny) for nx, ny, _, _ in mix]
    grids = _grids(mix)
    srv = trotter.Server(hbm_budget_bytes=8 << 30, max_slots=16, K=4, max_epoch_steps=12)
    try:
        tickets = [srv.submit(nx, ny, s, 0.05, theta, V, re, im)
                   for (nx, ny, theta, s), (re, im, V) in zip(mix, data)]
        got = []
        for t, (nx, ny, _, _) in zip(tickets, mix):
            assert srv.wait(t, 60000).status == 0
            got.append(srv.fetch(t, ny, nx, np.float32))
            srv.release(t)
        for g, (re, im, _), (*_, s), o in zip(grids, data, mix, got):
            g.set_state(re, im)
            g.evolve(s, 4)
            w = g.get_state(np.float32)
            assert np.array_equal(o[0], w[0]) and np.array_equal(o[1], w[1])
    finally:
        srv.close()
        for g in grids:
            g.close()


def test_angle_set_behind_another_streams_work():
    """The angle is set on a busy stream and again on the stream that evolves: what the
    batch reads must not be left to the busy stream's queue."""
    import torch
    nx, ny, theta, steps = 200, 90, 0.05, 9
    re, im, V = _inputs(nx, ny)
    busy, mine = torch.cuda.Stream(), torch.cuda.Stream()
    on_busy, on_mine = (trotter._VP(s.cuda_stream) for s in (busy, mine))
    grids = [trotter.Grid(nx, ny, "f32") for _ in range(2)]
    big = trotter.Grid(8192, 8192, "f32")
    try:
        big.set_potential(None, 0.05, 0.025)
        for g in grids:
            g.set_potential(V, 0.05, 0.01)
        trotter.evolve_batched(grids, [steps, steps])
        torch.cuda.synchronize()
        big.evolve(4000, stream=on_busy)                   # about 0.3 s
        grids[0].set_potential(V, 0.05, theta, on_busy)
        for g in grids:
            g.set_potential(V, 0.05, theta, on_mine)
            g.set_state(re, im, on_mine)
        trotter.evolve_batched(grids, [steps, steps], stream=on_mine)
        out = [torch.stack(g.get_state(np.float32, device=True, stream=on_mine)) for g in grids]
        assert not busy.query()
        torch.cuda.synchronize()
        grids[1].set_state(re, im)
        grids[1].evolve(steps)
        want = torch.stack(grids[1].get_state(np.float32, device=True))
        assert torch.equal(out[0], want) and torch.equal(out[1], want)
    finally:
        for g in grids + [big]:
            g.close()
