"""The calls this framework is used for, as cases that can be timed and checked.

Every case goes through the package's public entry points (`fdtd.Grid`,
`fdtd.Batch`, `fdtd.Adjoint`, `adjoint.beam_loss`) the way a program that
drives a Bessel-antenna run does: a box with its antenna (or the wall sheet) is
made once, and a pass advances it and reads the fields and the fluence back.
Sizes are those of the package's own workload recipes and of the tests.

  probe_48_f32        a script that watches a tiny box: two steps, then a look at everything (launches and latency)
  ring_64_f64         the small FP64 box with tangential injection that is run to compare implementations
  table1_b_f32        one of the paper's Table 1 boxes (20 cells per wavelength, odd width, no fluence)
  beam_256_f32        the reference beam in the configuration a grid has by default, with fluence
  beam_256_two_step   the same beam in the tuned configuration: two steps per launch, ranges balanced by measurement
  beam_256_f64        the same beam in FP64, the precision of the accuracy studies
  beam_512_f32        a wide box of the order / angle study, circular polarisation
  bessel_gauss_f32    Section 2's Bessel-Gauss box: z walls, CPML on all faces, the wall sheet (the largest box)
  sweep_f32           a sweep over cone angles and orders as one batch of uneven grids, 64 steps per call
  sweep_small_f32     a batch of small grids, with a remainder after the 64-step replay
  adjoint_f32         reverse-time steps with probe gradients, and the gradient of the antenna weights
  gradient_f32        one whole gradient of the beam loss: forward, checkpoints, replay and reverse

A state starts in mid-run: a few plane waves of the source wavelength with
random directions, amplitudes and polarisations under a window that vanishes
on the walls, and seeded antenna weights.
"""
import math

import numpy as np
import torch

EY = 1


# ---- the cases

def _dz(nz, dx, theta):
    """Cell size along z for whole axial periods, close to dx."""
    lam_z = 1.0 / math.cos(math.radians(theta))
    return max(1, round(nz * dx / lam_z)) * lam_z / nz


def _beam(name, nx, ny, nz, npml, per_lambda, theta, m, pol, radius, thick, steps, precision="f32", fluence=True,
          tile="default", inject="all"):
    case = dict(kind="beam", nx=nx, ny=ny, nz=nz, npml=npml, dx=1.0 / per_lambda,
                dz=_dz(nz, 1.0 / per_lambda, theta), theta=theta, m=m, pol=pol, radius=radius, thick=thick,
                steps=steps, precision=precision, fluence=fluence, tile=tile, inject=inject)
    if name:
        case["name"] = name
    return case


def _wall(name, nx, ny, nz, npml, npml_z, w0, steps, precision="f32", envelope="gauss"):
    case = dict(kind="wall", nx=nx, ny=ny, nz=nz, npml=npml, npml_z=npml_z, dx=0.05, dz=0.05, theta=25.0, w0=w0,
                plane=npml_z if npml_z else 1, steps=steps, precision=precision, fluence=True, envelope=envelope)
    if name:
        case["name"] = name
    return case


def _sweep(name, thetas, orders, steps, odd=0, precision="f32", nz=64):
    case = dict(kind="sweep", thetas=" ".join("%g" % t for t in thetas), orders=" ".join("%d" % m for m in orders),
                odd=odd, nz=nz, npml=16, dx=1.0 / 18, steps=steps, precision=precision)
    if name:
        case["name"] = name
    return case


def _reverse(name, n, ny, nz, steps, window, precision="f32"):
    theta, dx, npml = 15.0, 0.05, 16
    case = dict(kind="reverse", nx=n, ny=ny, nz=nz, npml=npml, dx=dx, dz=_dz(nz, dx, theta), theta=theta, m=0,
                pol="y", radius=0.8 * (min(n, ny) - 2 * npml) / 2.0, thick=3.0, steps=steps, window=window,
                precision=precision, fluence=False, tile="default", inject="all")
    if name:
        case["name"] = name
    return case


def _gradient(name, nx, ny, nz, steps, window, checkpoint, tile="two_step"):
    theta, dx, npml = 25.0, 1.0 / 16, 8
    case = dict(kind="gradient", nx=nx, ny=ny, nz=nz, npml=npml, dx=dx, dz=_dz(nz, dx, theta), theta=theta, m=0,
                pol="y", radius=0.6 * (min(nx, ny) - 2 * npml) / 2.0, thick=3.0, steps=steps, window=window,
                checkpoint=checkpoint, precision="f32", fluence=False, tile=tile, inject="all")
    if name:
        case["name"] = name
    return case


def listed():
    return [
        _beam("probe_48_f32", 48, 40, 16, 6, 16, 20.0, 0, "y", 10.0, 1.0, 2),
        _beam("ring_64_f64", 64, 64, 32, 8, 16, 20.0, 0, "x", 12.0, 1.0, 40, precision="f64", inject="tangential"),
        _beam("table1_b_f32", 332, 332, 46, 6, 20, 30.0, 1, "y", 149.0, 20.0, 40, fluence=False),
        _beam("beam_256_f32", 256, 256, 128, 16, 20, 10.0, 0, "y", 100.0, 1.0, 40),
        _beam("beam_256_two_step", 256, 256, 128, 16, 20, 10.0, 0, "y", 100.0, 1.0, 40, tile="two_step"),
        _beam("beam_256_f64", 256, 256, 128, 16, 20, 10.0, 0, "y", 100.0, 1.0, 10, precision="f64"),
        _beam("beam_512_f32", 512, 512, 64, 16, 24, 15.0, 1, "circ+", 192.0, 1.0, 21),
        _wall("bessel_gauss_f32", 411, 411, 738, 16, 16, 7.5, 10),
        _sweep("sweep_f32", (5, 10, 20, 30), (0, 1), 64),
        _sweep("sweep_small_f32", (30, 20), (0, 1, 2), 70),
        _reverse("adjoint_f32", 384, 384, 96, 100, 30),
        _gradient("gradient_f32", 160, 152, 40, 80, 20, 25),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["beam"] * 5 + ["wall"] * 2 + ["sweep", "reverse", "gradient"])
    if kind == "beam":
        precision = rng.choice(["f32", "f32", "f32", "f64"])
        nx, ny = _log(rng, 40, 560), _log(rng, 40, 560)
        if max(nx, ny) > 4 * min(nx, ny):
            nx = ny = max(nx, ny)
        nz = _log(rng, 5, 160)
        npml = rng.choice([6, 8, 10, 16])
        npml = min(npml, min(nx, ny) // 5)
        room = min(nx, ny) / 2.0 - npml - 2.0
        thick = min(rng.choice([1.0, 1.0, 3.0, 20.0]), room / 3.0)
        radius = rng.uniform(0.5, 0.95) * (room - thick / 2.0)
        cells = nx * ny * nz
        most = 3.0e8 if precision == "f32" else 6.0e7
        steps = max(1, min(rng.choice([1, 2, 7, 20, 41, 64]), int(most / cells)))
        tile = rng.choice(["default", "default", "two_step"]) if precision == "f32" else "default"
        return _beam(None, nx, ny, nz, npml, rng.choice([16, 20, 24]), rng.choice([10.0, 17.0, 25.0, 30.0]),
                     rng.choice([0, 1, 2, 3]), rng.choice(["y", "x", "circ+"]), round(radius, 3), round(thick, 3),
                     steps, precision, rng.choice([True, True, False]), tile, rng.choice(["all", "all", "tangential"]))
    if kind == "wall":
        precision = rng.choice(["f32", "f32", "f64"])
        nx, nz = _log(rng, 44, 411), _log(rng, 24, 738)
        ny = max(44, min(411, nx + rng.choice([-9, 0, 0, 5])))
        npml_z = min(rng.choice([0, 6, 16]), (nz - 2) // 2)
        most = 2.5e8 if precision == "f32" else 4.0e7
        steps = max(1, min(rng.choice([3, 10, 24]), int(most / (nx * ny * nz))))
        return _wall(None, nx, ny, nz, min(rng.choice([6, 16]), min(nx, ny) // 5), npml_z,
                     round(rng.uniform(0.5, 7.5), 3), steps, precision, rng.choice(["gauss", "cw"]))
    if kind == "sweep":
        thetas = rng.sample([7, 10, 15, 20, 25, 30], rng.choice([1, 2, 3]))
        return _sweep(None, thetas, rng.choice([(0,), (0, 1), (1, 3)]), rng.choice([5, 64, 67, 128]),
                      odd=rng.choice([0, 3, 13]), nz=_log(rng, 8, 64))
    if kind == "reverse":
        n = _log(rng, 80, 400)
        precision = rng.choice(["f32", "f32", "f64"])
        nz = _log(rng, 6, 96)
        steps = max(4, min(rng.choice([13, 40, 101]), int((1.5e9 if precision == "f32" else 2.0e8) / (n * n * nz))))
        return _reverse(None, n, n + rng.choice([0, 7]), nz, steps, rng.randint(2, steps), precision)
    n = _log(rng, 56, 200)
    return _gradient(None, n, n + rng.choice([-3, 0, 10]), _log(rng, 6, 40), rng.choice([30, 60, 80]),
                     rng.choice([10, 20]), rng.choice([16, 25]), rng.choice(["default", "two_step"]))


# ---- inputs

def _sweep_grids(case):
    """The grids of a sweep: N = 32 round(8 r0 / (32 dx)) cells across (plus `odd`), the ring at 0.8 of the interior."""
    out = []
    for theta in (float(t) for t in case["thetas"].split()):
        n = 32 * round(8 * 0.383 / math.sin(math.radians(theta)) / (32 * case["dx"])) + case["odd"]
        for m in (int(v) for v in case["orders"].split()):
            out.append(dict(kind="beam", nx=n, ny=n, nz=case["nz"], npml=case["npml"], dx=case["dx"],
                            dz=_dz(case["nz"], case["dx"], theta), theta=theta, m=m, pol="y",
                            radius=0.8 * (n - 2 * case["npml"]) / 2.0, thick=1.0, steps=case["steps"],
                            precision=case["precision"], fluence=True, tile="default", inject="all"))
    return out


def _dtype(case):
    return torch.float64 if case["precision"] == "f64" else torch.float32


def _initial(case, seed):
    """Six field arrays of a beam in mid-run, in the grid's precision."""
    g = np.random.default_rng(seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    waves = 5
    polar = g.uniform(0.1, 1.2, waves)
    azim = g.uniform(0, 2 * math.pi, waves)
    k = 2 * math.pi * np.stack([np.sin(polar) * np.cos(azim), np.sin(polar) * np.sin(azim), np.cos(polar)])
    amp = g.standard_normal((6, waves)) + 1j * g.standard_normal((6, waves))

    def axis(n, d, kk, window):
        p = np.arange(n)
        v = np.exp(1j * np.outer(kk, p * d))
        return torch.as_tensor(v * (np.sin(math.pi * p / n) if window else 1.0), device="cuda")

    walls = case["kind"] == "wall"
    X, Y = axis(nx, case["dx"], k[0], True), axis(ny, case["dx"], k[1], True)
    Z = axis(nz, case["dz"], k[2], walls)
    out = []
    for c in range(6):
        zy = torch.einsum("qk,qj->kjq", Z * torch.as_tensor(0.3 * amp[c], device="cuda")[:, None], Y).reshape(nz * ny, waves)
        left = torch.cat([zy.real, -zy.imag], dim=1)
        right = torch.cat([X.real, X.imag], dim=0)
        out.append((left @ right).reshape(nz, ny, nx).to(_dtype(case)))
        if c in (1, 2):       # tangential E on the walls
            out[c][:, :, 0] = 0
        if c in (0, 2):
            out[c][:, 0, :] = 0
        if walls and c < 2:
            out[c][0] = 0
    return out


def _weights(case, seed):
    g = np.random.default_rng(seed + 77)
    shape = (case["ny"], case["nx"])
    return 1.0 + 0.1 * g.standard_normal(shape), 0.1 * g.standard_normal(shape)


def _probes(case):
    """Cells within three central-lobe radii of the axis (inside the ring), on every plane."""
    r0 = 0.383 / math.sin(math.radians(case["theta"])) / case["dx"]
    i, j = np.arange(case["nx"])[None, :], np.arange(case["ny"])[:, None]
    r = np.hypot(i - case["nx"] / 2, j + 0.5 - case["ny"] / 2)
    cols = np.flatnonzero((r < min(case["radius"] - 2, 3 * r0)).ravel())
    return (np.arange(case["nz"])[:, None] * (case["nx"] * case["ny"]) + cols[None, :]).ravel()


def _loss_rows(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed + 5)
    n = _probes(case).size
    return torch.randn((case["window"], n), generator=g, device="cuda", dtype=torch.float64).to(_dtype(case))


def _target(case, seed):
    g = np.random.default_rng(seed + 9)
    return torch.as_tensor(0.5 + g.random(_probes(case).size), device="cuda")


def _ramp(case):
    return 1.0 if case["kind"] != "gradient" else 0.5


def _desc(fdtd, case):
    more = dict(z_walls=True, npml_z=case["npml_z"]) if case["kind"] == "wall" else {}
    return fdtd.make_grid_desc(case["nx"], case["ny"], case["nz"], case["npml"], case["dx"], case["dx"], case["dz"],
                               precision=case["precision"], fluence=case["fluence"], **more)


def _antenna(case):
    return dict(m=case["m"], theta=math.radians(case["theta"]), pol=case["pol"], r_center=case["radius"],
                thickness=case["thick"], ramp=_ramp(case), inject=case["inject"])


def _make_grid(fdtd, case, seed):
    grid = fdtd.Grid(_desc(fdtd, case))
    if case["kind"] == "wall":
        grid.set_wall_source(theta=math.radians(case["theta"]), w0=case["w0"], envelope=case["envelope"], ramp=1.0,
                             T=22.5, T0=45.0, plane=case["plane"])
    else:
        wa, wp = _weights(case, seed)
        grid.set_source(w_amp=wa, w_phase=wp, **_antenna(case))
        if case["tile"] == "two_step":
            grid.set_tile(7, 16, 2)
    for c, f in enumerate(_initial(case, seed)):
        grid.set_field(c, f)
    if case.get("tile") == "two_step":
        grid.measure_balance()
    return grid


def prepare(case, seed):
    from paper_2102_12978_gb300 import fdtd
    kind = case["kind"]
    if kind in ("beam", "wall"):
        return dict(kind=kind, grid=_make_grid(fdtd, case, seed), steps=case["steps"], fluence=case["fluence"])
    if kind == "sweep":
        grids = [_make_grid(fdtd, c, seed + 1000 * q) for q, c in enumerate(_sweep_grids(case))]
        return dict(kind=kind, grids=grids, batch=fdtd.Batch(grids), steps=case["steps"])
    if kind == "reverse":
        grid = _make_grid(fdtd, case, seed)
        grid.step(2)
        adj = fdtd.Adjoint(grid, EY, _probes(case))
        return dict(kind=kind, grid=grid, adj=adj, rows=_loss_rows(case, seed), steps=case["steps"],
                    window=case["window"])
    from paper_2102_12978_gb300 import adjoint
    problem = adjoint.BeamProblem(_desc(fdtd, case), _antenna(case), EY, _probes(case), _target(case, seed),
                                  case["steps"], case["window"], case["checkpoint"],
                                  tile=(7, 16, 1) if case["tile"] == "two_step" else None)
    problem.context()
    wa, wp = _weights(case, seed)
    return dict(kind=kind, problem=problem, wa=torch.as_tensor(wa), wp=torch.as_tensor(wp))


def _read(grid, fluence):
    out = dict(zip(("ex", "ey", "ez", "hx", "hy", "hz"), grid.fields()))
    if fluence:
        out["fluence"] = grid.fluence()
    return out


def run(state):
    kind = state["kind"]
    if kind in ("beam", "wall"):
        state["grid"].step(state["steps"])
        return _read(state["grid"], state["fluence"])
    if kind == "sweep":
        state["batch"].step(state["steps"])
        return [_read(g, True) for g in state["grids"]]
    if kind == "reverse":
        adj = state["adj"]
        adj.reset(state["steps"] + 40)          # the run's last step; the loss window is its latest states
        adj.step(state["window"], state["rows"])
        adj.step(state["steps"] - state["window"])
        ga, gp = adj.gradient()
        # H as one array: the probes read E_y, and the adjoint of H_y is then zero up to rounding
        return dict(e=[adj.field(c) for c in range(3)], h=torch.stack([adj.field(c) for c in range(3, 6)]),
                    d_amp=ga, d_phase=gp)
    from paper_2102_12978_gb300 import adjoint
    wa, wp = state["wa"].clone().requires_grad_(), state["wp"].clone().requires_grad_()
    loss = adjoint.beam_loss(wa, wp, state["problem"])
    loss.backward()
    return dict(loss=loss.detach(), d_amp=wa.grad, d_phase=wp.grad)


# ---- what a pass cannot do without

def _psi_values(case):
    """CPML values of one side (E or H): two components per shell and axis."""
    v = 2 * (2 * case["npml"]) * case["nz"] * (case["ny"] + case["nx"])
    if case["kind"] == "wall":
        v += 2 * (2 * case["npml_z"]) * case["ny"] * case["nx"]
    return v


def _work_of(case):
    """The state (fields, CPML values, fluence) in once and out once, the returned arrays written once; per step
    and cell the curl updates (2 x 18 operations) and the fluence term (33)."""
    cells, b = case["nx"] * case["ny"] * case["nz"], 8 if case["precision"] == "f64" else 4
    state = 6 * cells * b + 2 * _psi_values(case) * b + (8 * cells if case["fluence"] else 0)
    returned = 6 * cells * b + (8 * cells if case["fluence"] else 0)
    flops = case["steps"] * cells * (36 + (33 if case["fluence"] else 0))
    return 2 * state + returned, flops


def work(case):
    kind = case["kind"]
    if kind == "sweep":
        parts = [_work_of(c) for c in _sweep_grids(case)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    bytes_, flops = _work_of(case)
    cells = case["nx"] * case["ny"] * case["nz"]
    if kind == "reverse":       # the adjoint state starts at zero: written once, returned once; the loss rows read
        b = 8 if case["precision"] == "f64" else 4
        rows = case["window"] * _probes(case).size * b
        return {"bytes": 2 * 6 * cells * b + 2 * _psi_values(case) * b + rows + 16 * case["nx"] * case["ny"], "flops": flops}
    if kind == "gradient":      # forward, replay and reverse of every step; a checkpoint per segment written and read
        segments = -(-case["steps"] // case["checkpoint"])
        state = 6 * cells * 4 + 2 * _psi_values(case) * 4
        return {"bytes": 2 * segments * state, "flops": 3 * flops}
    return {"bytes": bytes_, "flops": flops}


# ---- the same in 64 bits, in plain torch

_HALF = ((0.5, 0.0, 0.0), (0.0, 0.5, 0.0), (0.0, 0.0, 0.5), (0.0, 0.5, 0.5), (0.5, 0.0, 0.5), (0.5, 0.5, 0.0))   # (x, y, z)


def _bessel(n, x):
    """J_n by its integral over a period; the trapezoid rule converges geometrically."""
    tau = 2 * math.pi * np.arange(1024) / 1024
    return np.mean(np.cos(n * tau[None, :] - x[:, None] * np.sin(tau)[None, :]), axis=1)


def _vector_beam(case, comp, x, y):
    """Complex amplitude of a component of the order-m TE beam of a transverse Hertz potential, without e^{i beta z}."""
    m, theta = case["m"], math.radians(case["theta"])
    k = 2 * math.pi
    K, beta = k * math.sin(theta), k * math.cos(theta)
    r, phi = np.hypot(x, y), np.arctan2(y, x)
    psi = {q: _bessel(m + q, K * r) * np.exp(1j * (m + q) * phi) for q in range(-2, 3)}
    # (d/dx + i d/dy) psi_q = -K psi_{q+1}, (d/dx - i d/dy) psi_q = K psi_{q-1}
    dx = {q: 0.5 * K * (psi[q - 1] - psi[q + 1]) for q in (-1, 0, 1)}
    dy = {q: 0.5j * K * (psi[q - 1] + psi[q + 1]) for q in (-1, 0, 1)}
    dxx = 0.5 * K * (dx[-1] - dx[1])
    dyy = 0.5j * K * (dy[-1] + dy[1])
    dxy = 0.5 * K * (dy[-1] - dy[1])
    p = psi[0]
    along_x = ([0 * p, 1j * beta * p, -dy[0]], [dxx + k * k * p, dxy, 1j * beta * dx[0]])     # curl and curl curl
    along_y = ([-1j * beta * p, 0 * p, dx[0]], [dxy, dyy + k * k * p, 1j * beta * dy[0]])
    if case["pol"] == "y":
        Q, R = along_x
    elif case["pol"] == "x":
        Q, R = along_y
    else:
        Q = [(a + 1j * b) / math.sqrt(2.0) for a, b in zip(along_x[0], along_y[0])]
        R = [(a + 1j * b) / math.sqrt(2.0) for a, b in zip(along_x[1], along_y[1])]
    v = [q / k for q in Q] if comp < 3 else [-1j * q / (k * k) for q in R]
    if case["inject"] == "tangential":
        c, s = x / r, y / r
        radial = c * v[0] + s * v[1]
        v = [v[0] - c * radial, v[1] - s * radial, v[2]]
    return v[comp % 3]


class _Yee:
    """The leapfrog with its CPML, antenna, wall sheet and fluence on whole FP64 arrays [z, y, x]."""

    def __init__(self, case):
        self.case = case
        self.walls = case["kind"] == "wall"
        self.d = (case["dz"], case["dx"], case["dx"])
        self.dt = 0.95 / math.sqrt(sum(1.0 / v ** 2 for v in self.d))
        n = (case["nz"], case["ny"], case["nx"])
        self.npml = (case["npml_z"] if self.walls else 0, case["npml"], case["npml"])
        self.prof = [[self._profile(n[a], self.npml[a], self.d[a], half, a) for half in (0, 1)] for a in range(3)]
        self.n = n
        self.points = None if self.walls else [self._points(c) for c in range(6)]
        if self.walls:
            i, j = np.arange(n[2])[None, :], np.arange(n[1])[:, None]
            r = np.hypot((i + 0.5 - n[2] / 2) * self.d[2], (j - n[1] / 2) * self.d[1])
            sheet = np.exp(-(r / case["w0"]) ** 2) * np.exp(-2j * math.pi * math.sin(math.radians(case["theta"])) * r)
            sheet[0] = 0.0
            self.sheet = torch.as_tensor(sheet, device="cuda")

    def _profile(self, n, npml, d, half, axis):
        if not npml:
            return None
        pos = np.arange(n) + 0.5 * half
        u = np.clip(np.where(pos < npml, npml - pos, np.where(pos > n - npml, pos - (n - npml), 0.0)) / npml, 0.0, None)
        sigma, alpha = 0.8 * 4.0 / d * u ** 3, 0.05 * 2 * math.pi * (1.0 - u)
        b = np.exp(-(sigma + alpha) * self.dt)
        a = np.where(sigma > 0, sigma * (b - 1.0) / np.maximum(sigma + alpha, 1e-300), 0.0)
        b, a = np.where(u > 0, b, 1.0), np.where(u > 0, a, 0.0)
        shape = [1, 1, 1]
        shape[axis] = npml
        cut = lambda v, lo: torch.as_tensor(v[:npml] if lo else v[n - npml:], device="cuda").reshape(shape)
        return [(cut(b, lo), cut(a, lo)) for lo in (True, False)]

    def _points(self, c):
        """Columns of a component's antenna points, their amplitudes and the z phases."""
        case, (nz, ny, nx) = self.case, self.n
        u = np.arange(nx)[None, :] + _HALF[c][0] - nx / 2
        v = np.arange(ny)[:, None] + _HALF[c][1] - ny / 2
        r2 = u * u + v * v
        lo, hi = case["radius"] - case["thick"] / 2, case["radius"] + case["thick"] / 2
        cols = np.flatnonzero(((r2 >= lo * lo) & (r2 < hi * hi)).ravel())
        jj, ii = np.divmod(cols, nx)
        amp = _vector_beam(case, c, u[0, ii] * case["dx"], v[jj, 0] * case["dx"])
        z = (np.arange(nz) + _HALF[c][2]) * case["dz"]
        phase = np.exp(2j * math.pi * math.cos(math.radians(case["theta"])) * z)
        return tuple(torch.as_tensor(t, device="cuda") for t in (cols, amp, phase))

    def zero_psi(self):
        """psi[side][k]: side 0 the E updates, 1 the H updates; k the six (field, axis) pairs, low and high shell."""
        out = []
        for _ in range(2):
            side = {}
            for f in range(3):
                for axis in range(3):
                    if axis == 2 - f or not self.npml[axis]:
                        continue
                    shape = list(self.n)
                    shape[axis] = self.npml[axis]
                    side[(f, axis)] = [torch.zeros(shape, dtype=torch.float64, device="cuda") for _ in range(2)]
            out.append(side)
        return out

    def _up(self, f, axis):
        if axis == 0 and not self.walls:
            return torch.roll(f, -1, 0)
        return torch.cat([f.narrow(axis, 1, f.shape[axis] - 1), torch.zeros_like(f.narrow(axis, 0, 1))], axis)

    def _down(self, f, axis):
        if axis == 0 and not self.walls:
            return torch.roll(f, 1, 0)
        return torch.cat([torch.zeros_like(f.narrow(axis, 0, 1)), f.narrow(axis, 0, f.shape[axis] - 1)], axis)

    def _slope(self, f, field, axis, side, psi):
        """df/daxis with the CPML of the shells; psi is replaced by its next value."""
        d = (self._up(f, axis) - f if side else f - self._down(f, axis)) / self.d[axis]
        prof = self.prof[axis][side]
        if prof is None:
            return d
        w, n = self.npml[axis], self.n[axis]
        (b0, a0), (b1, a1) = prof
        lo, hi = psi[side][(field, axis)]
        lo = b0 * lo + a0 * d.narrow(axis, 0, w)
        hi = b1 * hi + a1 * d.narrow(axis, n - w, w)
        psi[side][(field, axis)] = [lo, hi]
        return torch.cat([d.narrow(axis, 0, w) + lo, d.narrow(axis, w, n - 2 * w), d.narrow(axis, n - w, w) + hi], axis)

    def _time(self, t):
        case = self.case
        gauss = case.get("envelope") == "gauss"
        tp = t - 45.0 if gauss else t
        if gauss:
            f = math.exp(-((t - 45.0) / 22.5) ** 2)
        else:
            ramp = _ramp(case)
            f = math.sin(math.pi * t / (2 * ramp)) ** 2 if t < ramp else 1.0
        ph = 2 * math.pi * (tp - math.floor(tp))
        return complex(f * math.cos(ph), -f * math.sin(ph))

    def _add(self, fields, first, t, weights):
        for c in range(3):
            cols, amp, phase = self.points[first + c]
            w = amp * self._time(t)
            if weights is not None:
                wa, wp = weights
                w = w * torch.polar(wa.reshape(-1)[cols], wp.reshape(-1)[cols])
            s = torch.outer(phase.real, w.real) - torch.outer(phase.imag, w.imag)
            fields[c] = fields[c].reshape(self.n[0], -1).index_add(1, cols, s).reshape(self.n)

    def step(self, E, H, psi, step, weights, fluence=None):
        """One step; returns the new E, H and fluence (psi's lists are replaced in place)."""
        psi = [dict(psi[0]), dict(psi[1])]
        dt = self.dt
        s = lambda f, field, axis: self._slope(f, field, axis, 1, psi)
        new = [H[0] - dt * (s(E[2], 0, 1) - s(E[1], 0, 0)), H[1] - dt * (s(E[0], 1, 0) - s(E[2], 1, 2)),
               H[2] - dt * (s(E[1], 2, 2) - s(E[0], 2, 1))]
        if self.points:
            self._add(new, 3, (step + 0.5) * dt, weights)
        if fluence is not None:
            up = self._up
            ex = E[0] + up(E[0], 1)
            ey = E[1] + up(E[1], 2)
            ez = E[2] + up(E[2], 2)
            e = [0.25 * (ex + up(ex, 0)), 0.25 * (ey + up(ey, 0)), 0.25 * (ez + up(ez, 1))]
            h = [0.25 * (v + up(v, 2 - c)) for c, v in enumerate(a + b for a, b in zip(H, new))]
            fluence = fluence + dt * torch.sqrt((e[1] * h[2] - e[2] * h[1]) ** 2 + (e[2] * h[0] - e[0] * h[2]) ** 2
                                                + (e[0] * h[1] - e[1] * h[0]) ** 2)
        H = new
        s = lambda f, field, axis: self._slope(f, field, axis, 0, psi)
        E = [E[0] + dt * (s(H[2], 0, 1) - s(H[1], 0, 0)), E[1] + dt * (s(H[0], 1, 0) - s(H[2], 1, 2)),
             E[2] + dt * (s(H[1], 2, 2) - s(H[0], 2, 1))]
        if self.points:
            self._add(E, 0, (step + 1.0) * dt, weights)
        else:
            w = self.sheet * self._time((step + 1.0) * dt)
            k = self.case["plane"]
            E[0] = torch.cat([E[0][:k], E[0][k:k + 1] + w.real, E[0][k + 1:]], 0)
        clear = lambda f, axis: torch.cat([torch.zeros_like(f.narrow(axis, 0, 1)), f.narrow(axis, 1, f.shape[axis] - 1)], axis)
        E = [clear(E[0], 1), clear(E[1], 2), clear(clear(E[2], 2), 1)]
        if self.walls:
            E = [clear(E[0], 0), clear(E[1], 0), E[2]]
        return E, H, psi, fluence


def _exact_steps(case, seed):
    yee = _Yee(case)
    f = [t.double() for t in _initial(case, seed)]
    weights = None if yee.walls else tuple(torch.as_tensor(w, device="cuda") for w in _weights(case, seed))
    E, H, psi = f[:3], f[3:], yee.zero_psi()
    flu = torch.zeros(yee.n, dtype=torch.float64, device="cuda") if case["fluence"] else None
    with torch.no_grad():
        for n in range(case["steps"]):
            E, H, psi, flu = yee.step(E, H, psi, n, weights, flu)
    out = dict(zip(("ex", "ey", "ez", "hx", "hy", "hz"), E + H))
    if flu is not None:
        out["fluence"] = flu
    return out


def _flat(E, H, psi):
    return list(E) + list(H) + [t for side in psi for pair in side.values() for t in pair]


def _unflat(v, like):
    it = iter(v[6:])
    return v[:3], v[3:6], [{k: [next(it), next(it)] for k in side} for side in like]


def _exact_reverse(case, seed):
    """Each reverse step is the vector-Jacobian product of one step (linear in the state and in the source)."""
    yee = _Yee(case)
    like = yee.zero_psi()
    zeros = [torch.zeros(yee.n, dtype=torch.float64, device="cuda") for _ in range(6)]
    bar = _flat(zeros[:3], zeros[3:], like)
    wa, wp = (torch.as_tensor(w, device="cuda").requires_grad_() for w in _weights(case, seed))
    rows, cells = _loss_rows(case, seed).double(), torch.as_tensor(_probes(case), device="cuda")
    da, dp = torch.zeros_like(wa), torch.zeros_like(wp)
    end = case["steps"] + 40
    for r in range(case["steps"]):
        if r < case["window"]:
            bar[EY] = bar[EY].reshape(-1).index_add(0, cells, rows[r]).reshape(yee.n)
        x = [torch.zeros_like(t).requires_grad_() for t in bar]
        E, H, psi = _unflat(x, like)
        E, H, psi, _ = yee.step(E, H, psi, end - 1 - r, (wa, wp))
        y = _flat(E, H, psi)
        g = torch.autograd.grad(y, x + [wa, wp], [t.detach() for t in bar], allow_unused=True)
        bar = [torch.zeros_like(t) if v is None else v for v, t in zip(g, x)]
        da, dp = da + g[-2], dp + g[-1]
    return dict(e=bar[:3], h=torch.stack(bar[3:6]), d_amp=da.detach(), d_phase=dp.detach())


def _exact_gradient(case, seed):
    from torch.utils.checkpoint import checkpoint
    yee = _Yee(case)
    like = yee.zero_psi()
    wa, wp = (torch.as_tensor(w, device="cuda").requires_grad_() for w in _weights(case, seed))
    cells, target = torch.as_tensor(_probes(case), device="cuda"), _target(case, seed)
    zeros = [torch.zeros(yee.n, dtype=torch.float64, device="cuda") for _ in range(6)]
    v = _flat(zeros[:3], zeros[3:], like)
    total = 0.0

    def one(n, a, p, *x):
        E, H, psi = _unflat(list(x), like)
        E, H, psi, _ = yee.step(E, H, psi, n, (a, p))
        return tuple(_flat(E, H, psi))

    for n in range(case["steps"]):
        v = list(checkpoint(one, n, wa, wp, *v, use_reentrant=False))
        if n >= case["steps"] - case["window"]:
            total = total + v[EY].reshape(-1)[cells] ** 2
    loss = torch.linalg.norm(total / case["window"] - target) / torch.linalg.norm(target)
    loss.backward()
    return dict(loss=loss.detach(), d_amp=wa.grad.cpu(), d_phase=wp.grad.cpu())


def exact(case, seed):
    kind = case["kind"]
    if kind in ("beam", "wall"):
        return _exact_steps(case, seed)
    if kind == "sweep":
        return [_exact_steps(c, seed + 1000 * q) for q, c in enumerate(_sweep_grids(case))]
    return _exact_reverse(case, seed) if kind == "reverse" else _exact_gradient(case, seed)
