"""The work that programs give this framework, as cases that can be timed.

listed() names twelve cases over the whole range: one small evolution with its
report, FP64 and FP32 grids up to 8192 x 8192, ragged sides, the fourth-order
step, a time-dependent potential, a 3-D lattice, the gradient of the fidelity,
many grids at once and the request server.  draw() gives another case of the
same ranges.  prepare() makes a case's inputs on the GPU (host arrays for the
server) and the grid or server that a program keeps; run() is one pass through
the public entry points, from setting the state to reading it back; exact()
is the same result in plain torch FP64.
"""
import math

import numpy as np
import torch

from paper_1208_2407_gb300 import trotter

SERVE_SIDES = (128, 256, 512, 1024, 2048)
OBSERVABLES = ("norm", "x", "y", "x2", "y2", "e_kin", "e_pot")


def listed():
    return [
        # The smallest request of the serving mix: a short run on a 128 x 128
        # grid with a report first.  Latency and launches decide.
        dict(name="small_f32_128", kind="evolve", nx=128, ny=128, dtype="f32", steps=10,
             dt=0.05, theta=0.025, pot="gauss", report=True, table=False),
        # The plain validation workload: 256 x 256 in FP64, flat potential.
        dict(name="flat_f64_256", kind="evolve", nx=256, ny=256, dtype="f64", steps=100,
             dt=0.05, theta=0.025, pot="flat", report=False, table=False),
        # An ordinary study on a grid whose sides fit no tile.
        dict(name="ragged_f32_1001x777", kind="evolve", nx=1001, ny=777, dtype="f32", steps=150,
             dt=0.05, theta=0.025, pot="gauss", report=True, table=True),
        # The precision workload: a packet in a harmonic trap, 1000 steps.
        dict(name="trap_f32_2048", kind="evolve", nx=2048, ny=2048, dtype="f32", steps=1000,
             dt=0.05, theta=0.025, pot="trap", report=False, table=False),
        # The large grid of the throughput benchmark, everything included: the
        # state in, the table, the report, 200 steps, the state out.
        dict(name="large_f32_8192", kind="evolve", nx=8192, ny=8192, dtype="f32", steps=200,
             dt=0.05, theta=0.025, pot="gauss", report=True, table=True),
        # FP64 production at an ordinary, odd size.
        dict(name="ragged_f64_2047x1536", kind="evolve", nx=2047, ny=1536, dtype="f64", steps=40,
             dt=0.05, theta=0.025, pot="trap", report=True, table=True),
        # The fourth-order Suzuki step, for long steps at a given error.
        dict(name="order4_f32_4096", kind="order4", nx=4096, ny=4096, dtype="f32", steps=20,
             dt=0.1, theta=0.05, pot="gauss"),
        # A driven system: V0 + a(t) V1 with a field along x.
        dict(name="drive_f32_3000x2048", kind="drive", nx=3000, ny=2048, dtype="f32", steps=80,
             dt=0.05, theta=0.025, pot="trap"),
        # A packet in a 3-D trap.
        dict(name="trap3d_f32_256", kind="evolve3", nx=256, ny=256, nz=256, dtype="f32", steps=40,
             dt=0.05, theta=0.025, pot="trap"),
        # One step of fitting a potential: fidelity and its gradient.
        dict(name="adjoint_f32_1024", kind="adjoint", nx=1024, ny=1024, dtype="f32", steps=500,
             dt=0.05, theta=0.025, pot="trap", ckpt=50),
        # A sweep of independent grids of mixed sizes advanced together.
        dict(name="batch_f32_16", kind="batch", count=16, max_side=2048, max_steps=200,
             dt=0.05, theta=0.025, pot="gauss", mix=11),
        # The request server with host inputs, submitted at once.
        dict(name="serve_f32_16", kind="serve", count=16, max_side=1024, max_steps=500,
             dt=0.05, theta=0.025, pot="gauss", mix=12),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _side(rng, lo, hi):
    """A side, spread over the logarithm; about half are as drawn (odd ones
    among them), half the next multiple of 32."""
    n = _log_int(rng, lo, hi)
    return n if rng.random() < 0.5 else min(hi, (n + 31) // 32 * 32)


def _steps(rng, lo, hi, sites, most):
    """Steps in [lo, hi], at most `most` site-steps in all."""
    return max(1, min(_log_int(rng, lo, hi), int(most // sites)))


def draw(rng):
    kind = rng.choice(["f32", "f32", "f32", "f64", "order4", "drive", "evolve3", "adjoint",
                       "batch", "serve"])
    dt = math.exp(rng.uniform(math.log(0.02), math.log(0.1)))
    c = dict(dt=dt, theta=0.5 * dt, pot=rng.choice(["gauss", "trap"]))
    if kind in ("f32", "f64"):
        top = 8192 if kind == "f32" else 3000
        nx, ny = _side(rng, 96, top), _side(rng, 96, top)
        most, hi = (1.2e10, 1000) if kind == "f32" else (1.5e8, 120)
        c.update(kind="evolve", nx=nx, ny=ny, dtype=kind, steps=_steps(rng, 10, hi, nx * ny, most),
                 report=rng.random() < 0.5, table=rng.random() < 0.5)
        if rng.random() < 0.2:
            c["pot"] = "flat"
    elif kind in ("order4", "drive"):
        nx, ny = _side(rng, 256, 6000), _side(rng, 256, 6000)
        most = 8e8 if kind == "order4" else 2e9
        c.update(kind=kind, nx=nx, ny=ny, dtype="f32", steps=_steps(rng, 10, 200, nx * ny, most))
    elif kind == "evolve3":
        nx, ny, nz = (_side(rng, 64, 384) for _ in range(3))
        c.update(kind=kind, nx=nx, ny=ny, nz=nz, dtype="f32", pot="trap",
                 steps=_steps(rng, 10, 200, nx * ny * nz, 1e9))
    elif kind == "adjoint":
        nx, ny = _side(rng, 128, 2048), _side(rng, 128, 2048)
        c.update(kind=kind, nx=nx, ny=ny, dtype="f32", pot="trap", ckpt=rng.choice([25, 50, 64]),
                 steps=_steps(rng, 20, 500, nx * ny, 6e8))
    else:
        c.update(kind=kind, count=rng.randint(4, 24), mix=rng.randrange(1 << 20), pot="gauss",
                 max_side=2048 if kind == "batch" else 1024,
                 max_steps=200 if kind == "batch" else 500)
    return c


# --- inputs -----------------------------------------------------------------
def _rng(case, seed):
    return np.random.default_rng([seed, case["nx"], case["ny"], case.get("nz", 1)])


def _axis(n, centre, sigma, k, width=1.0):
    x = torch.arange(n, dtype=torch.float64, device="cuda")
    return torch.polar(torch.exp(-((x - centre) ** 2) / (4.0 * (width * sigma) ** 2)), k * x)


def _packet(axes):
    """The product of 1-D packets (x first), normalised, as FP64 (re, im)."""
    nrm = math.prod(float((a.abs() ** 2).sum()) for a in axes)
    psi = axes[0] / math.sqrt(nrm)
    for a in axes[1:]:
        psi = a.reshape((-1,) + (1,) * psi.dim()) * psi
    return psi.real.contiguous(), psi.imag.contiguous()


def _packet_params(r, sides):
    """A packet centred in the middle half, a few per cent of a side wide."""
    return [(r.uniform(n / 4.0, 3.0 * n / 4.0), r.uniform(min(16.0, n / 16.0), min(64.0, n / 8.0)),
             r.uniform(-1.0, 1.0)) for n in sides]


def _sides(case):
    return [case["nx"], case["ny"]] + ([case["nz"]] if "nz" in case else [])


def _potential(case, r):
    """FP64 potential of the grid's shape, or None for a flat one."""
    sides = _sides(case)
    if case["pot"] == "flat":
        return None
    if case["pot"] == "trap":
        w = 1e-2 if len(sides) == 3 else 1e-3
        V = torch.zeros((), dtype=torch.float64, device="cuda")
        for i, n in enumerate(sides):
            x = torch.arange(n, dtype=torch.float64, device="cuda") - n / 2.0
            V = V + (0.5 * w * w * x * x).reshape((-1,) + (1,) * i)
        return V.contiguous()
    nx, ny = sides
    cx, cy = r.uniform(0.0, nx, 32), r.uniform(0.0, ny, 32)
    amp, wid = r.uniform(-0.5, 0.5, 32), r.uniform(20.0, 200.0, 32)
    cx, cy, amp, wid = (torch.tensor(v, device="cuda")[:, None] for v in (cx, cy, amp, wid))
    x = torch.arange(nx, dtype=torch.float64, device="cuda")
    y = torch.arange(ny, dtype=torch.float64, device="cuda")
    gx = amp * torch.exp(-((x - cx) ** 2) / (2.0 * wid ** 2))
    gy = torch.exp(-((y - cy) ** 2) / (2.0 * wid ** 2))
    return gy.T @ gx


def _inputs(case, seed):
    """State (of the grid's type), potential and what the kind adds."""
    r = _rng(case, seed)
    params = _packet_params(r, _sides(case))
    re, im = _packet([_axis(n, *p) for n, p in zip(_sides(case), params)])
    td = torch.float64 if case["dtype"] == "f64" else torch.float32
    d = dict(re=re.to(td), im=im.to(td), V=_potential(case, r))
    if case["kind"] == "drive":
        # a field along x, oscillating in time, sampled at step midpoints
        x = torch.arange(case["nx"], dtype=torch.float64, device="cuda") - case["nx"] / 2.0
        d["V1"] = (x / case["nx"]).expand(case["ny"], case["nx"]).contiguous()
        t = (np.arange(case["steps"]) + 0.5) * case["dt"]
        d["a"] = r.uniform(0.5, 2.0) * np.sin(r.uniform(0.5, 3.0) * t + r.uniform(0.0, 6.0))
    if case["kind"] == "adjoint":
        # a target that the packet reaches: moved by its group velocity, a
        # little off and of another width
        T = case["steps"] * case["dt"]
        J = 2.0 * case["theta"] / case["dt"]
        wid = r.uniform(0.8, 1.25)
        axes = [_axis(n, c + 2.0 * J * math.sin(k) * T + r.uniform(-0.5, 0.5) * s, s, k, wid)
                for n, (c, s, k) in zip(_sides(case), params)]
        tre, tim = _packet(axes)
        d.update(tre=tre.to(td), tim=tim.to(td))
    return d


def _members(case):
    """The grids of a batch or of a serving mix, as cases of their own."""
    r = np.random.default_rng(case["mix"])
    sides = [s for s in SERVE_SIDES if s <= case["max_side"]]
    out = []
    for i in range(case["count"]):
        nx, ny = int(r.choice(sides)), int(r.choice(sides))
        if i % 4 == 3:                          # one in four fits no tile
            nx, ny = nx - int(r.integers(0, 64)), ny - int(r.integers(0, 64))
        out.append(dict(kind="evolve", nx=nx, ny=ny, dtype="f32", dt=case["dt"],
                        theta=case["theta"], pot=case["pot"],
                        steps=int(r.integers(10, case["max_steps"] + 1))))
    return out


def _grid(case, d):
    g = trotter.Grid(case["nx"], case["ny"], case["dtype"], nz=case.get("nz", 1))
    g.set_potential(d["V"], case["dt"], case["theta"], order=4 if case["kind"] == "order4" else 2)
    return g


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        ms = _members(case)
        ds = [_inputs(m, seed * 1000 + i) for i, m in enumerate(ms)]
        if kind == "batch":
            return dict(case=case, members=ms, inputs=ds, grids=[_grid(m, d) for m, d in zip(ms, ds)])
        ds = [{k: v.cpu().pin_memory() for k, v in d.items()} for d in ds]
        return dict(case=case, members=ms, inputs=ds,
                    server=trotter.Server(hbm_budget_bytes=8 << 30, max_slots=64))
    d = _inputs(case, seed)
    return dict(case=case, inputs=d, grid=_grid(case, d))


# --- one pass ---------------------------------------------------------------
def _read(case, g):
    return list(g.get_state(np.float64 if case["dtype"] == "f64" else np.float32, device=True))


def run(state):
    case, d = state["case"], state["inputs"]
    kind = case["kind"]
    if kind == "adjoint":
        # the optimiser has moved V: state and table anew, then the gradient
        g = state["grid"]
        g.set_state(d["re"], d["im"])
        g.set_potential(d["V"], case["dt"], case["theta"])
        F, grad = trotter.adjoint_fidelity_grad(g, d["tre"], d["tim"], case["steps"], case["ckpt"])
        return [grad]
    if kind == "batch":
        for g, x in zip(state["grids"], d):
            g.set_state(x["re"], x["im"])
        trotter.evolve_batched(state["grids"], [m["steps"] for m in state["members"]])
        return [_read(m, g) for m, g in zip(state["members"], state["grids"])]
    if kind == "serve":
        srv = state["server"]
        tickets = [srv.submit(m["nx"], m["ny"], m["steps"], m["dt"], m["theta"], x["V"], x["re"],
                              x["im"]) for m, x in zip(state["members"], d)]
        out = []
        for m, t in zip(state["members"], tickets):
            srv.wait(t)
            out.append(list(srv.fetch(t, m["ny"], m["nx"], np.float32)))
            srv.release(t)
        return out
    g = state["grid"]
    out = []
    g.set_state(d["re"], d["im"])
    if case.get("table"):
        g.set_potential(d["V"], case["dt"], case["theta"])
    if kind == "drive":
        g.set_drive(d["V1"], d["a"])
    if case.get("report"):
        o = g.observe()
        out.append({k: o[k] for k in OBSERVABLES})
    g.evolve(case["steps"])
    return out + _read(case, g)


def work(case):
    """Bytes: state in and out, potentials in, each once.  Flops: per site and
    step three merged sweeps per axis with one FMA per real component, and the
    phase's four FMAs."""
    kind = case["kind"]
    if kind in ("batch", "serve"):
        ws = [work(m) for m in _members(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    sides = _sides(case)
    sites, steps = math.prod(sides), case["steps"]
    es = 8 if case["dtype"] == "f64" else 4
    nbytes = 4 * es * sites + (2 * es * sites if case["pot"] != "flat" else 0)
    fma = 6 * len(sides) + 4
    if kind == "order4":
        fma *= 5
        nbytes += 2 * es * sites
    elif kind == "drive":
        fma += 12                              # sine and cosine of a_n dt V1, their rotation
        nbytes += es * sites
    elif kind == "adjoint":
        fma = 3 * fma + 4                      # psi forward; psi and lambda back; conj(lambda) psi
        nbytes += 4 * es * sites               # the target in, G out
    return {"bytes": nbytes, "flops": 2 * fma * sites * steps}


# --- the same in FP64 -------------------------------------------------------
def _sweep(psi, dim, parity, c, s):
    n = (psi.shape[dim] - parity) // 2
    if n < 1:
        return
    p = psi.narrow(dim, parity, 2 * n).unflatten(dim, (n, 2))
    a, b = p.select(dim + 1, 0), p.select(dim + 1, 1)
    a0 = a.clone()
    a.mul_(c).add_(b, alpha=1j * s)
    b.mul_(c).add_(a0, alpha=1j * s)


def _families(psi):
    """X-even, X-odd, Y-even, Y-odd[, Z-even, Z-odd]; x is the last axis."""
    return [(psi.dim() - 1 - ax, par) for ax in range(psi.dim()) for par in (0, 1)]


def _half(psi, theta, mirror):
    c, s = math.cos(theta), math.sin(theta)
    fam = _families(psi)
    for dim, par in (reversed(fam) if mirror else fam):
        _sweep(psi, dim, par, c, s)


def _step(psi, phase, theta):
    _half(psi, theta, False)
    if phase is not None:
        psi.mul_(phase)
    _half(psi, theta, True)


def _phase(V, dt):
    return None if V is None else torch.polar(torch.ones_like(V), -dt * V)


def _exact_state(case, d):
    psi = torch.complex(d["re"].double(), d["im"].double())
    dt, th, steps = case["dt"], case["theta"], case["steps"]
    if case["kind"] == "order4":
        p = 1.0 / (4.0 - 4.0 ** (1.0 / 3.0))
        w = [p, p, 1.0 - 4.0 * p, p, p]
        ph = {x: _phase(d["V"], x * dt) for x in set(w)}
        for _ in range(steps):
            for x in w:
                _step(psi, ph[x], x * th)
    elif case["kind"] == "drive":
        for n in range(steps):
            _step(psi, _phase(d["V"] + float(d["a"][n]) * d["V1"], dt), th)
    else:
        ph = _phase(d["V"], dt)
        for _ in range(steps):
            _step(psi, ph, th)
    return psi


def _exact_gradient(case, d):
    """dF/dV, F = |<phi|psi_T>|^2: psi and the costate step back together;
    each step adds 2 dt Im(conj(c) conj(lambda) psi) at its phase."""
    dt, th = case["dt"], case["theta"]
    V = d["V"]
    psi = _exact_state(case, d)
    lam = torch.complex(d["tre"].double(), d["tim"].double())
    c = torch.vdot(lam.flatten(), psi.flatten())
    back = _phase(V, -dt)
    G = torch.zeros_like(psi)
    for _ in range(case["steps"]):
        _half(psi, -th, False)
        _half(lam, -th, False)
        G += lam.conj() * psi
        psi.mul_(back)
        lam.mul_(back)
        _half(psi, -th, True)
        _half(lam, -th, True)
    return 2.0 * dt * (c.conj() * G).imag


def _exact_report(case, d):
    re, im = d["re"].double(), d["im"].double()
    p = re * re + im * im
    nrm = p.sum()
    x = torch.arange(case["nx"], dtype=torch.float64, device=p.device)
    y = torch.arange(case["ny"], dtype=torch.float64, device=p.device)
    px, py = p.sum(0), p.sum(1)
    J = 2.0 * case["theta"] / case["dt"]
    bonds = ((re[:, 1:] * re[:, :-1] + im[:, 1:] * im[:, :-1]).sum()
             + (re[1:] * re[:-1] + im[1:] * im[:-1]).sum())
    v = [nrm, (x * px).sum() / nrm, (y * py).sum() / nrm, (x * x * px).sum() / nrm,
         (y * y * py).sum() / nrm, -2.0 * J * bonds,
         (d["V"] * p).sum() if d["V"] is not None else torch.zeros(())]
    return {k: float(t) for k, t in zip(OBSERVABLES, v)}


def exact(case, seed):
    if case["kind"] in ("batch", "serve"):
        out = []
        for i, m in enumerate(_members(case)):
            psi = _exact_state(m, _inputs(m, seed * 1000 + i))
            out.append([psi.real.contiguous(), psi.imag.contiguous()])
        return out
    d = _inputs(case, seed)
    if case["kind"] == "adjoint":
        return [_exact_gradient(case, d)]
    out = [_exact_report(case, d)] if case.get("report") else []
    psi = _exact_state(case, d)
    return out + [psi.real.contiguous(), psi.imag.contiguous()]
