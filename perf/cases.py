"""The work a user of the solver has it do, as cases to measure.

A case is one call sequence of a user's program on prepared solvers: lattice
steps with the force history and the fields read back afterwards, step by step
with the force read after each step, a batch of solvers stepped as a sweep, the
two gradients of the hydrodynamic function, and the sine fit of a long force
history.  Sizes are those of the named workloads, the study, the tests and the
benchmark, or lie between them.

``exact`` restates the method in plain torch, in 64 bits, from the paper's
equations (full description in the comments of ``_Reference``); nothing of the
CUDA library is used there.
"""
from __future__ import annotations

import cmath
import functools
import math

import numpy as np
import torch

import inputs
from paper_2006_13631_gb300 import Solver, Sweep
from paper_2006_13631_gb300 import hlbm as api

_FLOAT = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
_NOISE = 1e-6  # density noise of the 4096^2 workload


# ------------------------------------------------------------------ the cases
def _flow(name, call, nx, ny, L, tau, n_sub, A, omega, steps, dtype, mesh, **more):
    """One solver (or several) of a lamina of chord L in an nx x ny lattice.

    mesh: (n_L, n_T, n_layers, h1, d_out) of inputs.lamina_mesh."""
    c = dict(name=name, call=call, nx=nx, ny=ny, L=L, T=L / 50.0, tau=tau, n_sub=n_sub, A=A, omega=omega, steps=steps,
             dtype=dtype, n_L=mesh[0], n_T=mesh[1], layers=mesh[2], h1=mesh[3], d_out=mesh[4], delta_f=2.0, bc="wall",
             levels=0, lumped=0, outer_fv=0)
    c.update(more)
    return c


def listed():
    cases = []
    hp = inputs.harmonic_params
    # A program coupled to the solver: every lattice step is a call of its own, followed by
    # a read of the force.  The ragged 203 x 157 lattice of the parity tests.
    A, om, tau = hp(24.0, 0.5, 100.0)
    cases.append(_flow("coupled-203x157-f32", "single", 203, 157, 24.0, tau, 24, A, om, 24, "f32", (60, 2, 12, 0.2, 4.0)))
    # A lamina on a spring and damper, moved by the fluid: the force of a step decides the next.
    cases.append(_flow("induced-512-f32", "steps", 512, 512, 32.0, 0.56, 50, 0.0, 0.0, 40, "f32",
                       (64, 2, 15, 0.25, 4.0), mass=0.25 * math.pi * 32.0 ** 2, period=400.0, y0=1.5))
    # A whole validation run in FP64: four periods, then the hydrodynamic function.
    A, om, tau = hp(20.0, 0.25, 500.0, tau=0.6)
    cases.append(_flow("theta-256-f64", "theta", 256, 256, 20.0, tau, 50, A, om, 96, "f64", (78, 2, 15, 0.25, 4.0)))
    # Reduced-precision lattice storage at 1024^2.
    A, om, tau = hp(32.0, 0.25, 500.0, tau=0.6)
    cases.append(_flow("steps-1024-f16", "steps", 1024, 1024, 32.0, tau, 50, A, om, 60, "f16", (64, 2, 15, 0.25, 4.0)))
    # The outer-node sums of the full update (an option of the Theta study), on a periodic box.
    A, om, tau = hp(48.0, 0.5, 200.0)
    cases.append(_flow("outerfv-769x640-f32", "steps", 769, 640, 48.0, tau, 50, A, om, 40, "f32",
                       (120, 2, 20, 0.2, 5.0), outer_fv=1, bc="periodic"))
    # The 4096^2 benchmark workload: the bandwidth-bound lattice beside a 200k-node patch.
    A, om, tau = hp(128.0, 1.0, 1000.0)
    big = (835, 10, 100, 0.1, 10.0)
    cases.append(_flow("steps-4096-f32", "steps", 4096, 4096, 128.0, tau, 64, A, om, 200, "f32", big, delta_f=3.0))
    # The same domain and patch on two levels with BF16 storage, and the paper's own set-up: chord
    # 800 on four levels (45k-node patch, n = 77), the run of its 35-point study.
    cases.append(_flow("levels2-1025-bf16", "steps", 1025, 1025, 128.0, tau, 64, A, om, 60, "bf16", big, delta_f=3.0,
                       levels=1))
    A, om, tau = hp(800.0, 2.0 * math.pi * 0.05, 100.0, tau=0.8)
    cases.append(_flow("study-800-levels4-f32", "steps", 1001, 401, 800.0, tau, 77, A, om, 120, "f32",
                       (1600, 2, 14, 0.2, 4.0), levels=3, T=8.0))
    # The parametric study as a sweep: six solvers of different chords and sub-step counts, packed.
    cases.append(dict(name="sweep-6-f32", call="sweep", count=6, L0=16.0, kc0=0.2, beta0=100.0, beta1=1500.0, steps=6,
                      dtype="f32"))
    # The gradient of Theta by central differences (seven solvers, created inside the call) and by the adjoint.
    A, om, tau = hp(20.0, 0.25, 500.0, tau=0.6)
    om *= 1.0131  # no node class changes within the quotient's step
    cases.append(_flow("gradient-256-f64", "gradient", 256, 256, 20.0, tau, 50, A, om, 48, "f64",
                       (78, 2, 15, 0.25, 4.0)))
    cases.append(_flow("adjoint-256-f64", "adjoint", 256, 256, 20.0, tau, 50, A, om, 48, "f64",
                       (78, 2, 15, 0.25, 4.0)))
    # The smallest call: the sine fit of a force history already on the device (20 periods of 5120 steps).
    cases.append(dict(name="fit-102400", call="fit", samples=102400, period=5120.3, dtype="f64"))
    return cases


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _min_edge(L, T, n_L, n_T, h1):
    # the corner arcs of the first layer have two segments over a quarter circle of radius h1
    return min(2.0 * h1 * math.sin(math.pi / 8.0), L / n_L, T / n_T)


def draw(rng):
    call = rng.choice(["steps"] * 8 + ["single", "single", "theta", "sweep", "gradient", "adjoint", "fit"])
    if call == "fit":
        n = int(_log(rng, 500, 400000))
        return dict(call="fit", samples=n, period=n / rng.uniform(3.0, 30.0), dtype="f64")
    if call == "sweep":
        b0 = _log(rng, 100.0, 300.0)
        return dict(call="sweep", count=rng.randint(3, 7), L0=rng.choice([16.0, 20.0, 24.0]), kc0=_log(rng, 0.1, 0.4),
                    beta0=b0, beta1=b0 * _log(rng, 3.0, 12.0), steps=rng.randint(2, 6), dtype="f32")
    small = call in ("gradient", "adjoint")
    dtype = "f64" if small else rng.choice(["f32", "f32", "f32", "f64", "f16", "bf16"])
    L = round(_log(rng, 16.0, 24.0 if small else 40.0 if dtype == "f64" or call != "steps" else 128.0), 1)
    T = L / rng.choice([50.0, 100.0])
    d_out = rng.choice([4.0, 4.0, 5.0, 6.5])
    layers = rng.randint(10, 16) if small else int(_log(rng, 10, 30 if dtype == "f64" else 50))
    layers = min(layers, int(d_out / 0.15))  # the layers grow outwards from h1
    h1 = round(max(0.1, min(0.3, 0.7 * d_out / layers)), 3)
    n_L = int(L * rng.uniform(1.8, 2.5 if small else 5.0))
    n_T = 2
    if small:  # a whole number of periods, few steps: the test's own regime
        kc, beta = rng.uniform(0.2, 0.3), rng.uniform(400.0, 600.0)
        A, om, tau = inputs.harmonic_params(L, kc, beta, tau=0.6)
        steps = int(math.ceil(1.76 * 2.0 * math.pi / om)) + 1
    else:
        for _ in range(100):
            kc, beta, vmax = _log(rng, 0.15, 1.0), _log(rng, 30.0, 1000.0), rng.uniform(0.015, 0.025)
            A, om, tau = inputs.harmonic_params(L, kc, beta, vmax=vmax)
            if 0.507 <= tau <= 0.75:
                break
        steps = int(_log(rng, 12, 60))
    h = _min_edge(L, T, n_L, n_T, h1)
    tau_u = tau - 0.5
    n_sub = max(rng.randint(20, 40), math.ceil(1.0 / (1.9 * tau_u)), math.ceil(6.0 * tau_u / (h * h)))
    while small and n_sub * steps * n_L * layers > 50 * 48 * 78 * 15:  # no costlier than the listed ones
        om *= 1.1
        steps = int(math.ceil(1.76 * 2.0 * math.pi / om)) + 1
    levels = rng.choice([0, 0, 0, 1, 3]) if call == "steps" else 0
    span = int(2 * A + 2 * d_out + T + 24)
    if levels:
        nx, ny = int(L * rng.uniform(1.5, 3.0) + span) | 1, int(L * rng.uniform(0.5, 2.0) + span) | 1
    else:
        w = _log(rng, 4.0, 10.0 if small else 32.0)
        nx, ny = min(4096, int(w * L)), min(4096, int(w * L * rng.uniform(0.6, 1.0)) + span)
    if call == "theta":
        steps = min(400, int(math.ceil(2.0 * math.pi / om)) + 2)
    # as much work as the largest listed case at most
    cost = nx * ny + 60.0 * n_sub * n_L * 2.0 * layers
    steps = max(4, min(steps, int(3.0e9 / cost))) if not small and call != "theta" else steps
    c = _flow(None, call, nx, ny, L, tau, n_sub, A, om, steps, dtype, (n_L, n_T, layers, h1, d_out),
              bc=rng.choice(["wall", "wall", "periodic"]), levels=levels, T=T)
    del c["name"]
    if not small:
        c["lumped"] = int(rng.random() < 0.15)
        c["outer_fv"] = int(rng.random() < 0.12)
        if call == "single" and rng.random() < 0.4:  # as the lamina moved by the fluid
            c.update(A=0.0, omega=0.0, mass=0.25 * math.pi * L * L * rng.uniform(1.0, 3.0),
                     period=round(rng.uniform(300.0, 900.0), 1), y0=round(rng.uniform(0.5, 1.5), 2))
    return c


# ------------------------------------------------------------ building inputs
@functools.lru_cache(maxsize=32)
def _mesh(L, T, n_L, n_T, layers, h1, d_out):
    return inputs.lamina_mesh(L, T, n_L, n_T, layers, h1, d_out)


def _mesh_of(w):
    m = w.mesh_args
    return _mesh(w.L, w.T, m["n_L"], m["n_T"], m["n_layers"], m["h1"], m["d_out"])


def _level_sizes(nx, ny, count):
    """(nx, ny, ox, oy) of count coarser levels, each a box centred in the next
    (odd sizes for the inner ones), about 1.6, 1.5 and 1.25 times as wide."""
    out = []
    for k in range(count):
        grow = 1.6 if k == 0 else 1.5 if k == 1 else 1.25
        half = ((nx + 1) // 2, (ny + 1) // 2)
        size = [max(int(grow * h), h + 8) for h in half]
        if k + 1 < count:
            size = [s | 1 for s in size]
        out.append((size[0], size[1], (size[0] - half[0]) // 2, (size[1] - half[1]) // 2))
        nx, ny = size
    return out


def _workloads(case):
    """inputs.Workload of each solver of a case."""
    if case["call"] == "sweep":
        out = []
        n = case["count"]
        for k in range(n):
            beta = case["beta0"] * (case["beta1"] / case["beta0"]) ** (k / max(1, n - 1))
            L = case["L0"] * 2 ** (2 * k // n)
            A, om, tau = inputs.harmonic_params(L, case["kc0"] * (1.0 + 0.5 * (k % 2)), beta)
            spacing = 0.2 if k % 2 else 0.3
            layers = int(round(4.0 / spacing)) + 1
            mesh = dict(n_L=int(L / spacing), n_T=2, n_layers=layers, h1=4.0 / (layers - 1), d_out=4.0)
            h = _min_edge(L, L / 50.0, mesh["n_L"], 2, mesh["h1"])
            n_sub = max(20, math.ceil(1.0 / (1.9 * (tau - 0.5))), math.ceil(6.0 * (tau - 0.5) / (h * h)))
            side = int(32 * L)
            out.append(inputs.Workload(f"sweep-{k}", side, side, L, L / 50.0, 0.5 * side + 0.3, 0.5 * side + 0.2, tau,
                                       n_sub, inputs.MOTION_HARMONIC, A=A, omega=om, dtype=case["dtype"],
                                       noise_amp=_NOISE, mesh_args=mesh))
        return out
    nx, ny, bc = case["nx"], case["ny"], case["bc"]
    w = inputs.Workload(case["call"], nx, ny, case["L"], case["T"], 0.5 * nx + 0.3, 0.5 * ny + 0.2, case["tau"],
                        case["n_sub"], inputs.MOTION_HARMONIC, A=case["A"], omega=case["omega"],
                        delta_f=case["delta_f"], dtype=case["dtype"], lumped=case["lumped"],
                        outer_fv=case["outer_fv"], noise_amp=_NOISE,
                        mesh_args=dict(n_L=case["n_L"], n_T=case["n_T"], n_layers=case["layers"], h1=case["h1"],
                                       d_out=case["d_out"]))
    if bc == "periodic":
        w.bc_x = w.bc_y = inputs.BC_PERIODIC
    if "mass" in case:
        w.motion, w.mass, w.y0 = inputs.MOTION_INDUCED, case["mass"], case["y0"]
        w.stiffness = case["mass"] * (2.0 * math.pi / case["period"]) ** 2
    w.levels = _level_sizes(nx, ny, case["levels"])
    return [w]


def _density(w, seed):
    """Initial densities of the lattice and of its coarser levels."""
    lev = [inputs.initial_density(l[0], l[1], w.rho0, w.noise_amp, seed + 101 * (k + 1)) for k, l in enumerate(w.levels)]
    return inputs.initial_density(w.nx, w.ny, w.rho0, w.noise_amp, seed), lev


def _history(case, seed):
    """A force history [n + 1][2] of a harmonically moved lamina: carrier, third harmonic, noise."""
    g = np.random.default_rng(seed)
    t = np.arange(case["samples"] + 1, dtype=np.float64)
    om = 2.0 * math.pi / case["period"]
    amp, ph = g.uniform(0.5, 1.5), g.uniform(0.0, 2.0 * math.pi)
    fy = amp * np.sin(om * t + ph) + 0.05 * amp * np.sin(3.0 * om * t) + 0.02 * g.standard_normal(t.size)
    return np.stack([0.1 * g.standard_normal(t.size), fy], axis=1), om


def _fit_weights():
    return 1.0, 0.5  # dL/d(Re Theta), dL/d(Im Theta) of the adjoint's objective


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = case
    if case["call"] == "fit":
        f, s.omega = _history(case, seed)
        s.force = torch.from_numpy(f).cuda()
        return s
    s.work = _workloads(case)
    if case["call"] in ("gradient", "adjoint"):  # the call creates its solvers itself
        w = s.work[0]
        s.inputs = api.workload_inputs(w, _mesh_of(w), _density(w, seed)[0])
        return s
    s.solvers = []
    for k, w in enumerate(s.work):
        rho, lev = _density(w, seed + 1000 * k)
        s.solvers.append(Solver(w, mesh=_mesh_of(w), rho_init=rho, level_rho_init=lev or None))
    s.time = 0
    s.last = [None] * len(s.solvers)
    if case["call"] == "sweep":
        s.sweep = Sweep(s.solvers)
        s.sweep.pack()
    return s


# ------------------------------------------------------------------- one pass
def _as(x, dtype):
    """Host results, which the library gives in FP64, in the precision they were computed in."""
    return torch.from_numpy(x).to(_FLOAT[dtype])


def _near(w):
    """The rows and columns the lamina and its fictitious curve stay within."""
    ax, ay = 0.5 * w.L + w.delta_f + 2.0, 0.5 * w.T + w.delta_f + max(w.A, abs(w.y0)) + 2.0
    return (slice(max(0, int(w.yc - ay)), int(w.yc + ay) + 2), slice(max(0, int(w.xc - ax)), int(w.xc + ax) + 2))


def _rest_inside(w, cls, rho, ux, uy):
    """Nodes that are not discretization nodes carry no field: density rho0 at rest."""
    box = _near(w)
    off = cls[box] != 0
    rho[box][off], ux[box][off], uy[box][off] = w.rho0, 0.0, 0.0


def _read(s, k, force):
    """Force since the pass began, node classes, lattice, level and patch fields of solver k."""
    w, sol, dt = s.work[k], s.solvers[k], s.case["dtype"]
    rho, ux, uy, pr, pu, pv = sol.fields()
    cls = sol.struct_class()
    _rest_inside(w, cls, rho, ux, uy)
    out = dict(force=_as(force, dt), cls=cls, rho=_as(rho, dt), ux=_as(ux, dt), uy=_as(uy, dt),
               patch_rho=_as(pr, dt), patch_ux=_as(pu, dt), patch_uy=_as(pv, dt))
    for q in range(len(w.levels)):
        for n, v in zip(("rho", "ux", "uy"), sol.level_macro(q + 1)):
            out[f"level{q + 1}_{n}"] = _as(v, dt)
    return out


def run(s):
    c = s.case
    call = c["call"]
    if call == "fit":
        return list(api.hlbm_fit_static(s.force.data_ptr() + 8, 2, 0, c["samples"], s.omega,
                                        torch.cuda.current_stream().cuda_stream))
    if call == "gradient":
        grid, patch, motion = s.inputs
        th, g, _ = api.hlbm_theta_gradient(grid, patch, c["tau"], motion, c["steps"], 0.5, 1.25)
        # a difference quotient of values exact to 1e-13 over steps of 1e-4 carries single precision
        return dict(theta=np.array([th.real, th.imag]), grad=g.astype(np.complex64))
    if call == "adjoint":
        grid, patch, motion = s.inputs
        th, g, _, _ = api.hlbm_theta_adjoint(grid, patch, c["tau"], motion, c["steps"], 0.5, 1.25, *_fit_weights(), 16)
        return dict(theta=np.array([th.real, th.imag]), grad=g)
    n = c["steps"]
    t0 = s.time
    if call == "sweep":
        s.sweep.step(n)
        s.time += n
        out = []
        for k, sol in enumerate(s.solvers):
            fx, fy = api.hlbm_force(sol.h, t0 + 1, n)
            _, _, _, pr, pu, pv = sol.fields()
            out.append(dict(force=_as(np.stack([fx, fy], 1), c["dtype"]), patch_rho=_as(pr, c["dtype"]),
                            patch_ux=_as(pu, c["dtype"]), patch_uy=_as(pv, c["dtype"])))
        return out
    sol = s.solvers[0]
    if call == "single":
        fx, fy = np.empty(n), np.empty(n)
        for k in range(n):
            sol.step(1)
            fx[k: k + 1], fy[k: k + 1] = api.hlbm_force(sol.h, t0 + k + 1, 1)
    else:
        sol.step(n)
        fx, fy = api.hlbm_force(sol.h, t0 + 1, n)
    s.time += n
    out = _read(s, 0, np.stack([fx, fy], 1))
    if call == "theta":
        out["theta"] = _as(np.array(sol.gamma(*_theta_window(c))), c["dtype"])
    return out


def _theta_window(c):
    periods = c["steps"] * c["omega"] / (2.0 * math.pi)
    return (1.0, 3.0) if periods >= 3.9999 else (0.1 * periods, 0.8 * periods)


# ------------------------------------------------------------------------ work
def _one_step(w, elem):
    """Bytes and flops of a lattice step: every population read and written once per level
    step, the patch's populations and geometry once, 36 flops per FV row entry and sub-step
    (seven entries a row), about 130 per lattice node."""
    lat = w.nx * w.ny + sum(l[0] * l[1] / 2.0 ** (k + 1) for k, l in enumerate(w.levels))
    m = _mesh_of(w)
    pe = 8 if elem == 8 else 4
    return 18.0 * elem * lat + (28 * pe + 100) * m.n_nodes, 130.0 * lat + 36.0 * 7.0 * m.n_nodes * w.n_sub


def work(case):
    if case["call"] == "fit":
        n = case["samples"] + 1
        return {"bytes": 8.0 * n, "flops": 60.0 * n}
    elem = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}[case["dtype"]]
    b = f = 0.0
    for w in _workloads(case):
        sb, sf = _one_step(w, elem)
        b += sb * case["steps"]
        f += sf * case["steps"]
        if case["call"] not in ("gradient", "adjoint"):
            b += 24.0 * (w.nx * w.ny + sum(l[0] * l[1] for l in w.levels) + _mesh_of(w).n_nodes)
    if case["call"] == "gradient":
        b, f = 7.0 * b, 7.0 * f
    if case["call"] == "adjoint":  # forward, forward again, and a reverse of about twice the work
        b, f = 4.0 * b, 4.0 * f
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------- the exact values
_CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
_CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
_OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
_W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


class _Reference:
    """The method in plain torch, FP64 (or complex128: every decision is taken on real parts, so
    that an imaginary step of a parameter gives the derivative with the decisions held fixed).

    Populations are held as f - w rho0.  Patch arrays are [n, 9], lattice arrays [9, ny, nx].
    One step: relocate and refill the patch, classify, feed the lattice interpolation nodes,
    stream-collide (and couple the levels), feed the outer patch nodes, n_sub FV sub-steps,
    force on the lamina."""

    def __init__(self, w, mesh, rho, lev_rho, A=None, omega=None, tau=None, dtype=torch.float64):
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.ct, self.w = dtype, w
        self.A = w.A if A is None else A
        self.omega = w.omega if omega is None else omega
        self.tau = w.tau_s if tau is None else tau
        self.t, self.r0 = 0, w.rho0
        R = self.real
        self.cx, self.cy, self.wt = R(_CX), R(_CY), R(_W)
        self._patch_tables(mesh)
        self._wall_tables(mesh)
        # lattice and levels at equilibrium at rest
        self.cls = self.win = None
        self.f = self._rest(rho)
        self.pre = self.f.clone()
        self.taus = [0.5 + (self.tau - 0.5) / 2 ** k for k in range(len(w.levels) + 1)]
        self.lev = [[self._rest(r), None] for r in lev_rho]  # current and next buffer of each coarser level
        self.Y, self.V = (w.y0, w.v0) if w.motion == inputs.MOTION_INDUCED else (self._y(0), 0.0)
        self.Yprev = self.Y
        c = self._centre(self.Y)
        self._classify(c)
        for k in range(len(self.lev)):
            self._couple(k, 0, initial=True)
        self.P = self._from_lattice(self._bilinear(self.pre, self.xy[:, 0] + c[0], self.xy[:, 1] + c[1]))
        self.force = [self._force()]

    # ---- small helpers
    def real(self, x):
        return torch.as_tensor(np.asarray(x), dtype=torch.float64, device=self.dev)

    def num(self, x):
        return torch.as_tensor(x, dtype=self.ct, device=self.dev)

    def _rest(self, rho):
        r = self.real(rho) - self.r0
        return (self.wt[:, None, None] * r).to(self.ct)

    def _y(self, t):
        s = cmath.sin(self.omega * t) if self.ct.is_complex else math.sin(self.omega * t)
        return self.A * s

    def _centre(self, Y):
        return self.w.xc, self.w.yc + Y

    def _moments(self, f):  # [..., 9] -> drho, ux, uy
        dr = f.sum(-1)
        rho = self.r0 + dr
        return dr, (f @ self.cx.to(self.ct)) / rho, (f @ self.cy.to(self.ct)) / rho

    def _feq(self, dr, ux, uy):
        cu = ux[..., None] * self.cx + uy[..., None] * self.cy
        usq = (ux * ux + uy * uy)[..., None]
        return self.wt * (dr[..., None] + (self.r0 + dr)[..., None] * (3 * cu + 4.5 * cu * cu - 1.5 * usq))

    def _state(self, f):  # drho, ux, uy, f^neq stacked: what the interpolations carry
        dr, ux, uy = self._moments(f)
        return torch.cat([torch.stack([dr, ux, uy], -1), f - self._feq(dr, ux, uy)], -1)

    def _rebuild(self, st, k):
        return self._feq(st[..., 0], st[..., 1], st[..., 2]) + k * st[..., 3:]

    def _from_lattice(self, st):
        return self._rebuild(st, 1 - 1 / (2 * self.tau))

    def _bilinear(self, box, x, y):
        ix, iy = torch.floor(x.real).long(), torch.floor(y.real).long()
        ax, ay = x - ix, y - iy
        st = 0
        for q, wq in enumerate(((1 - ax) * (1 - ay), ax * (1 - ay), (1 - ax) * ay, ax * ay)):
            st = st + wq[:, None] * self._state(box[:, iy + (q >> 1), ix + (q & 1)].T)
        return st

    # ---- patch geometry: FV rows on median-dual control volumes, wall edges
    def _patch_tables(self, mesh):
        xy, tri, kind = np.asarray(mesh.xy, np.float64), np.asarray(mesh.tri, np.int64), np.asarray(mesh.kind)
        n = len(xy)
        X, Y = xy[tri, 0], xy[tri, 1]
        a2 = (X[:, 1] - X[:, 0]) * (Y[:, 2] - Y[:, 0]) - (X[:, 2] - X[:, 0]) * (Y[:, 1] - Y[:, 0])
        area = 0.5 * np.abs(a2)
        gx = np.stack([(Y[:, (j + 1) % 3] - Y[:, (j + 2) % 3]) / a2 for j in range(3)], 1)
        gy = np.stack([(X[:, (j + 2) % 3] - X[:, (j + 1) % 3]) / a2 for j in range(3)], 1)
        vol = np.zeros(n)
        np.add.at(vol, tri.ravel(), np.repeat(area / 3.0, 3))
        key, vx, vy, vc = [], [], [], []
        for p in range(3):
            for k in range(3):
                key.append(tri[:, p] * n + tri[:, k])
                vx.append(-area / 3.0 * gx[:, k])
                vy.append(-area / 3.0 * gy[:, k])
                vc.append(area * (11.0 / 54.0 if p == k else 7.0 / 108.0))
        u, inv = np.unique(np.concatenate(key), return_inverse=True)
        val = np.zeros((3, len(u)))
        for row, v in zip(val, (vx, vy, vc)):
            np.add.at(row, inv, np.concatenate(v))
        P, K = u // n, u % n
        val /= vol[P]
        if self.w.lumped:
            val[2] = (P == K)
        first = np.searchsorted(P, np.arange(n + 1))
        width = int(np.diff(first).max())
        slot = np.arange(len(u)) - first[P]
        nb = np.repeat(np.arange(n)[:, None], width, 1)
        m = np.zeros((3, n, width))
        nb[P, slot] = K
        m[:, P, slot] = val
        self.nb = torch.as_tensor(nb, device=self.dev)
        self.mat = self.real(m).permute(1, 0, 2).contiguous().to(self.ct)  # [n, 3, width]
        self.xy, self.kind = self.real(xy), torch.as_tensor(kind, device=self.dev)
        self.wall = torch.nonzero(self.kind == inputs.KIND_WALL)[:, 0]
        self.outer = torch.nonzero(self.kind == inputs.KIND_OUTER)[:, 0]
        # triangles: vertex a and the gradients of the barycentric coordinates; each node's star
        self.tri = torch.as_tensor(tri, device=self.dev)
        self.ta, self.gx, self.gy = self.real(np.stack([X[:, 0], Y[:, 0]], 1)), self.real(gx), self.real(gy)
        order = np.argsort(tri.ravel(), kind="stable")
        start = np.searchsorted(tri.ravel()[order], np.arange(n + 1))
        star = np.repeat((order[start[:-1]] // 3)[:, None], int(np.diff(start).max()), 1)
        for j in range(star.shape[1]):
            has = start[:-1] + j < start[1:]
            star[has, j] = order[(start[:-1] + j)[has]] // 3
        self.star = torch.as_tensor(star, device=self.dev)
        # triangles that can hold a lattice node near the fictitious curve
        qx = np.maximum(np.abs(X.mean(1)) - 0.5 * self.w.L, 0.0)
        qy = np.maximum(np.abs(Y.mean(1)) - 0.5 * self.w.T, 0.0)
        far = np.hypot(qx, qy) - self.w.delta_f
        self.band = torch.as_tensor(np.nonzero((far > -3.0) & (far < 2.0))[0], device=self.dev)

    def _wall_tables(self, mesh):
        tri, kind, xy = np.asarray(mesh.tri, np.int64), np.asarray(mesh.kind), np.asarray(mesh.xy)
        a, b = tri[:, (0, 1, 2)].ravel(), tri[:, (1, 2, 0)].ravel()
        lo, hi = np.minimum(a, b), np.maximum(a, b)
        _, inv, count = np.unique(lo * len(xy) + hi, return_inverse=True, return_counts=True)
        edge = (count[inv] == 1) & (kind[a] == inputs.KIND_WALL) & (kind[b] == inputs.KIND_WALL)
        a, b = a[edge], b[edge]
        e = xy[b] - xy[a]
        self.sa, self.sb = (torch.as_tensor(v, device=self.dev) for v in (a, b))
        self.sn = self.real(np.stack([-e[:, 1], e[:, 0]], 1)).to(self.ct)  # towards the fluid, times the length

    def _coords(self, k, x, y):  # barycentric coordinates of (x, y) in triangles k
        px, py = x - self.ta[k, 0], y - self.ta[k, 1]
        lb = self.gx[k, 1] * px + self.gy[k, 1] * py
        lc = self.gx[k, 2] * px + self.gy[k, 2] * py
        return torch.stack([1 - lb - lc, lb, lc], -1)

    # ---- one step
    def _refill(self, dY):
        # a relocated node lies in its own star or in those of its neighbours, inside the body,
        # or outside the patch: a step moves it by a fraction of an element
        x, y = self.xy[:, 0].to(self.ct), self.xy[:, 1] + dY
        low = self._coords(self.star, x.real[:, None], y.real[:, None]).amin(-1)
        best, at = low.max(1)
        k = self.star.gather(1, at[:, None])[:, 0]
        o = torch.nonzero(best < -1e-12)[:, 0]
        if len(o):
            wide = self.star[self.tri[self.star[o]]].reshape(len(o), -1)
            best[o], at = self._coords(wide, x.real[o, None], y.real[o, None]).amin(-1).max(1)
            k[o] = wide.gather(1, at[:, None])[:, 0]
        lam = self._coords(k, x, y).to(self.ct)
        new = (lam[:, :, None] * self.P[self.tri[k]]).sum(1)
        out = best < -1e-12
        body = out & (x.real.abs() <= 0.5 * self.w.L) & (y.real.abs() <= 0.5 * self.w.T)
        keep = body | (self.kind == inputs.KIND_WALL)
        new[keep] = self.P[keep]
        o = torch.nonzero(out & ~keep)[:, 0]
        if len(o):
            c = self._centre(self.Y)
            new[o] = self._from_lattice(self._bilinear(self.pre, self.xy[o, 0] + c[0], self.xy[o, 1] + c[1]))
        self.P = new

    def _inside(self, x, y, c):
        qx = ((x - c[0]).abs() - 0.5 * self.w.L).clamp(min=0.0)
        qy = ((y - (c[1].real if isinstance(c[1], complex) else c[1])).abs() - 0.5 * self.w.T).clamp(min=0.0)
        return qx * qx + qy * qy < self.w.delta_f ** 2

    def _classify(self, c):
        cy = c[1].real if isinstance(c[1], complex) else c[1]
        rx, ry = 0.5 * self.w.L + self.w.delta_f + 3, 0.5 * self.w.T + self.w.delta_f + 4
        x0, y0 = int(math.floor(c[0] - rx)), int(math.floor(cy - ry))
        nx, ny = int(2 * rx) + 3, int(2 * ry) + 3
        x = torch.arange(x0 - 1, x0 + nx + 1, device=self.dev, dtype=torch.float64)[None, :]
        y = torch.arange(y0 - 1, y0 + ny + 1, device=self.dev, dtype=torch.float64)[:, None]
        ins = self._inside(x, y, c)
        mid = ins[1:-1, 1:-1]
        disc = torch.zeros_like(mid)
        for i in range(1, 9):
            disc |= ~ins[1 + _CY[i]: 1 + _CY[i] + ny, 1 + _CX[i]: 1 + _CX[i] + nx]
        self.cls_prev, self.win_prev = self.cls, self.win
        self.cls = mid.to(torch.int8) * (2 - (mid & disc).to(torch.int8))  # 0 disc, 1 interpolation, 2 unused
        self.win = (x0, y0, nx, ny)

    def _class_map(self, cls, win):
        out = torch.zeros((self.w.ny, self.w.nx), dtype=torch.int8, device=self.dev)
        out[win[1]: win[1] + win[3], win[0]: win[0] + win[2]] = cls
        return out

    def _fill(self, c):
        x0, y0, nx, ny = self.win
        need = self.cls == 1
        if self.cls_prev is not None:  # nodes that have just become discretization nodes too
            px, py = self.win_prev[0], self.win_prev[1]
            xa, xb = max(x0, px), min(x0 + nx, px + self.win_prev[2])
            ya, yb = max(y0, py), min(y0 + ny, py + self.win_prev[3])
            was = torch.zeros_like(need)
            was[ya - y0: yb - y0, xa - x0: xb - x0] = self.cls_prev[ya - py: yb - py, xa - px: xb - px] != 0
            need = need | ((self.cls == 0) & was)
        at = torch.nonzero(need)
        y, x = at[:, 0] + y0, at[:, 1] + x0
        qx, qy = (x.double() - c[0]).to(self.ct), y.double() - c[1]
        k = torch.empty(len(x), dtype=torch.long, device=self.dev)
        for a in range(0, len(x), 256):
            s = slice(a, a + 256)
            low = self._coords(self.band[None, :], qx.real[s, None], qy.real[s, None]).amin(-1)
            k[s] = self.band[low.argmax(1)]
        lam = self._coords(k, qx, qy).to(self.ct)
        st = (lam[:, :, None] * self._state(self.P[self.tri[k]])).sum(1)
        self.f[:, y, x] = self._rebuild(st, 2 * (self.tau - 1) / (2 * self.tau - 1)).T

    def _pull(self, f, bcx, bcy):
        ny, nx = f.shape[1:]
        out = torch.empty_like(f)
        for i in range(9):
            src, cx, cy = f[i], _CX[i], _CY[i]
            g = torch.roll(src, (cy, cx), (0, 1))
            row, col = (0 if cy > 0 else ny - 1), (0 if cx > 0 else nx - 1)
            if cy and bcy == inputs.BC_OUTFLOW:
                g[row] = torch.roll(src[row], cx, 0)
            if cx and bcx == inputs.BC_OUTFLOW:
                g[:, col] = torch.roll(src[:, col], cy, 0)
                if cy and bcy == inputs.BC_OUTFLOW:
                    g[row, col] = src[row, col]
            if cy and bcy == inputs.BC_WALL:
                g[row] = f[_OPP[i]][row]
            if cx and bcx == inputs.BC_WALL:
                g[:, col] = f[_OPP[i]][:, col]
            out[i] = g
        return out

    def _collide(self, f, tau):
        dr = f.sum(0)
        rho = self.r0 + dr
        ux = (f[1] - f[3] + f[5] - f[6] - f[7] + f[8]) / rho
        uy = (f[2] - f[4] + f[5] + f[6] - f[7] - f[8]) / rho
        usq = 1.5 * (ux * ux + uy * uy)
        out = torch.empty_like(f)
        for i in range(9):
            cu = _CX[i] * ux + _CY[i] * uy
            out[i] = f[i] - (f[i] - _W[i] * (dr + rho * (3 * cu + 4.5 * cu * cu - usq))) / tau
        return out

    def _couple(self, k, t1, initial=False):
        """Level k restricts onto level k + 1 when it has caught up with it, and rebuilds its ring from it."""
        if not initial and t1 % (1 << k):
            return
        fine = self.f if k == 0 else self.lev[k - 1][0]
        coarse = self.lev[k]
        nxc, nyc, ox, oy = self.w.levels[k]
        nx, ny = fine.shape[2], fine.shape[1]
        tf, tc = self.taus[k], self.taus[k + 1]
        if initial or t1 % (2 << k) == 0:
            dst = coarse[0] if initial else coarse[1]
            sub = fine[:, 2: ny - 2: 2, 2: nx - 2: 2]
            st = self._state(sub.permute(1, 2, 0))
            val = self._rebuild(st, 2 * (tc - 1) / (tf - 1)).permute(2, 0, 1).clone()
            if k == 0:  # nothing retained reads the nodes under the lamina
                val[:, self._class_map(self.cls, self.win)[2: ny - 2: 2, 2: nx - 2: 2] != 0] = 0.0
            dst[:, oy + 1: oy + (ny - 1) // 2, ox + 1: ox + (nx - 1) // 2] = val
            if not initial:
                self.lev[k] = coarse = [coarse[1], coarse[0]]
        bufs = [coarse[0]] + ([coarse[1]] if not initial and (t1 >> k) & 1 else [])
        half = ((nx + 1) // 2, (ny + 1) // 2)
        for axis, edges in ((0, (0, ny - 1)), (1, (0, nx - 1))):
            for e in edges:
                line = 0
                for b in bufs:
                    if axis == 0:
                        src = b[:, oy + e // 2, ox - 1: ox + half[0] + 1]
                    else:
                        src = b[:, oy - 1: oy + half[1] + 1, ox + e // 2]
                    line = line + self._state(src.T) / len(bufs)
                n = nx if axis == 0 else ny
                st = torch.empty((n, 12), dtype=self.ct, device=self.dev)
                st[0::2] = line[1:-1]
                st[1::2] = (9 * (line[1:-2] + line[2:-1]) - (line[:-3] + line[3:])) / 16
                ring = self._rebuild(st, (tf - 1) / (2 * (tc - 1))).T
                if axis == 0:
                    fine[:, e, :] = ring
                else:
                    fine[:, 1:-1, e] = ring[:, 1:-1]

    def _fv_sums(self, f):  # dt_u times the right-hand side, all rows
        dr, ux, uy = self._moments(f)
        both = torch.cat([f, f - self._feq(dr, ux, uy)], 1)[self.nb]  # [n, width, 18]
        s = torch.bmm(self.mat, both)  # rows: g_x, g_y, C
        return (s[:, 0, :9] * self.cx + s[:, 1, :9] * self.cy - s[:, 2, 9:] / (self.tau - 0.5)) / self.w.n_sub

    def _wall_speed(self, theta, v1):
        if self.w.motion == inputs.MOTION_INDUCED:
            return self.V + theta * (v1 - self.V)
        a = self.omega * (self.t + theta)
        return self.A * self.omega * (cmath.cos(a) if self.ct.is_complex else math.cos(a))

    def step(self):
        w, t = self.w, self.t
        v1 = y1 = None
        if w.motion == inputs.MOTION_INDUCED:
            v1 = self.V + (float(self.force[-1][1]) - w.damping * self.V - w.stiffness * self.Y) / w.mass
            y1 = self.Y + v1
        else:
            self.Y = self._y(t)
        c = self._centre(self.Y)
        if t > 0:
            self._refill(self.Y - self.Yprev)
            self._classify(c)
        self._fill(c)
        for k in range(len(self.lev), 0, -1):
            if t % (1 << k) == 0:
                last = k == len(self.lev)
                bc = (w.bc_x, w.bc_y) if last else (inputs.BC_OUTFLOW, inputs.BC_OUTFLOW)
                self.lev[k - 1][1] = self._collide(self._pull(self.lev[k - 1][0], *bc), self.taus[k])
        bc = (w.bc_x, w.bc_y) if not self.lev else (inputs.BC_OUTFLOW, inputs.BC_OUTFLOW)
        pre = self._pull(self.f, *bc)
        self.f = self._collide(pre, self.tau)
        x0, y0, nx, ny = self.win
        box = self.f[:, y0: y0 + ny, x0: x0 + nx]
        box[:, self.cls == 2] = 0.0  # never read
        for k in range(len(self.lev)):
            self._couple(k, t + 1)
        ox, oy = self.xy[self.outer, 0] + c[0], self.xy[self.outer, 1] + c[1]
        s0, s1 = self._bilinear(self.pre, ox, oy), self._bilinear(pre, ox, oy)
        self.pre = pre
        zero = torch.zeros((), dtype=self.ct, device=self.dev)
        for m in range(w.n_sub):
            th = (m + 1) / w.n_sub
            new = self.P + self._fv_sums(self.P)
            dr, ux, uy = self._moments(new[self.wall])
            V = self.num(self._wall_speed(th, v1))
            new[self.wall] += self._feq(dr, zero.expand_as(dr), V.expand_as(dr)) - self._feq(dr, ux, uy)
            star = self._from_lattice((1 - th) * s0 + th * s1)
            if w.outer_fv:
                mixed = self.P.clone()
                mixed[self.outer] = star
                star = star + self._fv_sums(mixed)[self.outer]
            new[self.outer] = star
            self.P = new
        self.force.append(self._force())
        self.Yprev = self.Y
        if w.motion == inputs.MOTION_INDUCED:
            self.Y, self.V = y1, v1
        self.t = t + 1

    def _force(self):
        if not len(self.sa):
            return torch.zeros(2, dtype=self.ct, device=self.dev)

        def stress(p):
            f = self.P[p]
            dr, ux, uy = self._moments(f)
            q = f - self._feq(dr, ux, uy)
            cx, cy = self.cx.to(self.ct), self.cy.to(self.ct)
            return -dr / 3 - q @ (cx * cx), -(q @ (cx * cy)), -dr / 3 - q @ (cy * cy)

        s = [0.5 * (a + b) for a, b in zip(stress(self.sa), stress(self.sb))]
        return torch.stack([(s[0] * self.sn[:, 0] + s[1] * self.sn[:, 1]).sum(),
                            (s[1] * self.sn[:, 0] + s[2] * self.sn[:, 1]).sum()])

    # ---- read-back
    def fields(self):
        f = self.f.permute(1, 2, 0)
        dr, ux, uy = self._moments(f)
        cls = self._class_map(self.cls, self.win)
        for v in (dr, ux, uy):
            v[cls != 0] = 0.0
        return cls, self.r0 + dr, ux, uy

    def theta(self, discard, fit):
        T = 2.0 * math.pi / (self.omega.real if isinstance(self.omega, complex) else self.omega)
        return self.theta_over(math.ceil(discard * T), math.floor((discard + fit) * T))

    def theta_over(self, t0, t1):
        F = torch.stack([f[1] for f in self.force[t0: t1 + 1]])
        a, b, rms = _sine_fit(F, t0, self.num(self.omega))
        N = 0.25 * math.pi * self.r0 * self.omega ** 2 * self.w.L ** 2 * self.A
        return a / N, b / N, rms / abs(N)


def _sine_fit(F, t0, omega):
    t = torch.arange(t0, t0 + len(F), dtype=torch.float64, device=F.device)
    s, c = torch.sin(omega * t), torch.cos(omega * t)
    ss, sc, cc, fs, fc = (s * s).sum(), (s * c).sum(), (c * c).sum(), (F * s).sum(), (F * c).sum()
    det = ss * cc - sc * sc
    a, b = (fs * cc - fc * sc) / det, (fc * ss - fs * sc) / det
    e = F - (a * s + b * c)
    return a, b, ((e * e).real.mean() if e.is_complex() else (e * e).mean()).sqrt()


def _run_reference(w, seed, steps, **at):
    rho, lev = _density(w, seed)
    r = _Reference(w, _mesh_of(w), rho, lev, **at)
    for _ in range(steps):
        r.step()
    return r


def exact(case, seed):
    call, n = case["call"], case["steps"] if "steps" in case else 0
    if call == "fit":
        f, om = _history(case, seed)
        return [float(v) for v in _sine_fit(torch.from_numpy(f[:, 1].copy()), 0, om)]
    work_ = _workloads(case)
    if call in ("gradient", "adjoint"):
        w = work_[0]
        T = 2.0 * math.pi / w.omega
        win = (math.ceil(0.5 * T), math.floor(1.75 * T))
        if call == "gradient":
            base = dict(A=w.A, omega=w.omega, tau=w.tau_s)
            th = [float(v) for v in _run_reference(w, seed, n).theta_over(*win)[:2]]
            grad = []
            for k, v in base.items():
                ends = []
                for sign in (-1.0, 1.0):
                    r = _run_reference(w, seed, n, **{k: v + sign * 1e-4 * v})
                    re, im, _ = r.theta_over(*win)
                    ends.append(complex(float(re), float(im)))
                grad.append((ends[1] - ends[0]) / (2e-4 * v))
            return dict(theta=np.array(th), grad=np.array(grad).astype(np.complex128))
        wre, wim = _fit_weights()
        grad, th = [], None
        for k, v in dict(A=w.A, omega=w.omega, tau=w.tau_s).items():
            r = _run_reference(w, seed, n, dtype=torch.complex128, **{k: complex(v, 1e-30 * v)})
            re, im, _ = r.theta_over(*win)
            th = [float(re.real), float(im.real)]
            grad.append(float((wre * re + wim * im).imag) / (1e-30 * v))
        return dict(theta=np.array(th), grad=np.array(grad))
    out = []
    for k, w in enumerate(work_):
        r = _run_reference(w, seed + 1000 * k, n)
        pr, pu, pv = r._moments(r.P)
        o = dict(force=torch.stack(r.force[1:]), patch_rho=r.r0 + pr, patch_ux=pu, patch_uy=pv)
        if call == "sweep":
            out.append(o)
            continue
        cls, rho, ux, uy = r.fields()
        o.update(cls=cls, rho=rho, ux=ux, uy=uy)
        for q, (cur, _) in enumerate(r.lev):
            d, a, b = r._moments(cur.permute(1, 2, 0))
            o.update({f"level{q + 1}_rho": r.r0 + d, f"level{q + 1}_ux": a, f"level{q + 1}_uy": b})
        if call == "theta":
            o["theta"] = torch.stack([v.reshape(()) for v in r.theta(*_theta_window(case))])
        out.append(o)
    return out if call == "sweep" else out[0]
