"""The work that users of the library have it do, as a list of measurable cases.

A case is one simulation job on a lattice (kind "job": set the initial fields,
advance a number of iterations, write the fields) or one batch of requests
through the serving loop (kind "serve").  Sizes, materials, loads and
precisions are those of the repository's benchmark configurations and of the
paper's examples, from a 40 x 40 lattice, whose iterations are pure latency,
to the 16384 x 16384 one, which fills the memory bus.
"""
import math

import numpy as np
import torch

from paper_2502_00920_gb300 import inputs as I
from paper_2502_00920_gb300 import lbs

DEVICE = "cuda"


def _job(name, load, nx, ny, steps, precision, model="nh", nu=0.2, tau=0.55, extrap="own"):
    c = dict(kind="job", load=load, nx=nx, ny=ny, steps=steps, precision=precision, model=model, nu=nu, tau=tau,
             extrap=extrap)
    return dict(c, name=name) if name else c


def _serve(name, requests, trace, max_nx, max_ny, max_steps):
    c = dict(kind="serve", requests=requests, trace=trace, max_nx=max_nx, max_ny=max_ny, max_steps=max_steps,
             precision="fp32")
    return dict(c, name=name) if name else c


def listed():
    return [
        # the paper's simple-shear example at its own size and length (t = 2.2): the smallest job users run
        _job("shear_40_svk_fp64", "paper_shear", 40, 40, 98, "fp64", "svk"),
        # uniaxial tension on the benchmark's 32 x 32 block in single precision: many iterations of a tiny lattice
        _job("tension_32_nh_fp32", "tension", 32, 32, 400, "fp32"),
        # the paper's bending wave, the whole history (t = 12) of its 4:1 beam in double precision
        _job("wave_160x40_nh_fp64", "paper_wave", 160, 40, 537, "fp64"),
        # one run of the 256 x 256 shear sweep, in each storage precision
        _job("shear_256_svk_fp32", "shear", 256, 256, 500, "fp32", "svk"),
        _job("shear_256_svk_fp64", "shear", 256, 256, 200, "fp64", "svk"),
        # an odd-sized block with the two-point wall extrapolation and the linear comparison material
        _job("pull_391x173_le_fp32_linear", "tension", 391, 173, 150, "fp32", "le", extrap="linear"),
        # a ragged plate under a tip pulse in half-precision storage
        _job("pulse_1021x509_svk_fp16s", "cantilever", 1021, 509, 300, "fp16s", "svk"),
        # the long beam of the cantilever configuration
        _job("cantilever_4096x256_nh_fp32", "cantilever", 4096, 256, 500, "fp32", nu=0.25),
        # the periodic wave field on a large lattice in double precision
        _job("waves_4096_nh_fp64", "periodic", 4096, 4096, 40, "fp64", nu=0.3),
        # the largest lattice of the benchmark, single precision and half-precision storage
        _job("waves_16384_nh_fp32", "periodic", 16384, 16384, 100, "fp32", nu=0.3),
        _job("waves_16384_nh_fp16s", "periodic", 16384, 16384, 100, "fp16s", nu=0.3),
        # a batch of mixed requests through the server, submitted at once
        _serve("serve_10_mixed_fp32", 10, 4, 1024, 512, 240),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    if rng.random() < 0.12:
        return _serve(None, rng.randint(4, 10), rng.randint(0, 10 ** 6), _log_int(rng, 128, 1024),
                      _log_int(rng, 64, 512), rng.randint(120, 240))
    precision = rng.choice(["fp64", "fp32", "fp32", "fp16s"])
    model = rng.choice(["nh", "nh", "svk", "svk", "le"])
    load = rng.choice(["tension", "shear", "cantilever", "paper_shear", "paper_wave", "periodic", "periodic"])
    if load in ("cantilever", "paper_wave") and model == "svk":
        model = "nh"  # (the paper bends neo-Hooke beams; SVK blocks give way under the tip traction)
    # node updates of one job, bounded by what the precision's throughput allows in a tenth of a second or two
    updates = {"fp64": 3e8, "fp32": 3e9, "fp16s": 3e9}[precision]
    nx, ny = _log_int(rng, 32, 6000), _log_int(rng, 32, 6000)
    while nx * ny * 20 > updates:
        nx, ny = _log_int(rng, 32, 6000), _log_int(rng, 32, 6000)
    steps = max(20, min(rng.randint(40, 500), int(updates / (nx * ny))))
    if load in ("cantilever", "paper_wave") and ny > nx:
        nx, ny = ny, nx  # beams lie along x
    extrap = "linear" if load not in ("periodic", "paper_wave") and rng.random() < 0.2 else "own"
    # histories stay within the horizon in which the scheme's walls are stable
    if load != "periodic":
        steps = min(steps, 120 if extrap == "linear" else 300)
    # periodic fields carry nu = 0.3 (neutral there); walls amplify above 1/4 and at low nu
    nu = 0.3 if load == "periodic" else round(rng.uniform(0.15, 0.25), 3)
    return _job(None, load, nx, ny, steps, precision, model, nu, round(rng.uniform(0.55, 0.6), 3), extrap)


# ------------------------------------------------------------------ inputs
def _sim_case(c):
    """The library's description of a job."""
    load, nx, ny, steps = c["load"], c["nx"], c["ny"], c["steps"]
    if load == "tension":
        s = I.tension(nx, ny, steps, ramp=200, peak=0.05)
    elif load == "shear":
        s = I.shear(ny, steps, gamma=0.5, ramp=20000).replace(nx=nx)
    elif load == "cantilever":
        s = I.cantilever(nx, ny, steps, width=200, amp=0.05)
    elif load == "paper_shear":
        s = I.paper_shear(c["model"], c["nu"], ny).replace(nx=nx)
    elif load == "paper_wave":
        s = I.paper_wave(c["tau"], ny).replace(nx=nx)
    else:
        s = I.roofline(ny, steps, nx=nx)
    return s.replace(model=c["model"], nu=c["nu"], tau=c["tau"], precision=c["precision"], extrap=c["extrap"])


def _initial(c, s, seed):
    """Seeded smooth initial displacement and velocity on the device: the
    repository's random field on periodic lattices, a few low Fourier modes
    of small strain where there are walls."""
    if c["load"] == "periodic":
        corr = max(8.0, min(64.0, min(s.nx, s.ny) / 8))
        s = s.replace(seed=seed, init_args=dict(corr=corr, modes=64, strain=0.2))
        return None, I.grf_velocity(s, device=DEVICE)
    rng = np.random.default_rng(seed)
    x = torch.arange(s.nx, dtype=torch.float64, device=DEVICE) / s.nx
    y = torch.arange(s.ny, dtype=torch.float64, device=DEVICE) / s.ny
    fields = []
    for amp in (1e-3 * min(1.0, s.nx / s.ny), 1e-2):  # (strains stay small on narrow lattices)
        f = torch.zeros((s.ny, s.nx, 2), dtype=torch.float64, device=DEVICE)
        for a in range(2):
            for _ in range(3):
                kx, ky = rng.integers(1, 3, 2)
                ph, w = rng.uniform(0, 2 * math.pi, 2), rng.uniform(0.5, 1.0)
                f[:, :, a] += w * amp * torch.outer(torch.cos(2 * math.pi * int(ky) * y + ph[1]),
                                                    torch.sin(2 * math.pi * int(kx) * x + ph[0]))
        fields.append(f)
    return tuple(fields)


def _requests(c, seed):
    """The requests of a batch: the repository's serving trace at the case's
    sizes (its Poisson ratios folded into the range in which every load stays
    finite), load amplitudes drawn from the seed."""
    rng = np.random.default_rng(seed)
    out = []
    for _, r in I.serving_trace(c["requests"], seed=c["trace"], max_nx=c["max_nx"], max_ny=c["max_ny"], min_steps=100,
                                max_steps=c["max_steps"], precision=c["precision"]):
        k = float(rng.uniform(0.5, 1.0))
        edges = tuple(I.Edge(e.kind, e.shape, (k * e.amp[0], k * e.amp[1]), e.t0, e.t1, e.s, e.unit) for e in r.edges)
        # a displacement ramp keeps the pace of the trace's long histories
        edges = tuple(I.Edge(e.kind, e.shape, (0.02 * e.amp[0], e.amp[1]), e.t0, e.t1, e.s, e.unit)
                      if e.shape == "disp_ramp" else e for e in edges)
        out.append(r.replace(nu=0.1 + r.nu / 3, edges=edges))
    return out


def prepare(case, seed):
    if case["kind"] == "serve":
        return dict(kind="serve", server=lbs.Server(precision=case["precision"]), requests=_requests(case, seed))
    s = _sim_case(case)
    u0, v0 = _initial(case, s, seed)
    sim = lbs.Simulation(s)
    shape = (s.ny, s.nx, 2)
    out = [torch.empty(shape, dtype=torch.float64, device=DEVICE) for _ in range(2)]
    # P of the largest lattices stays where it is: their users take u and v out
    out.append(torch.empty(shape[:2] + (4,), dtype=torch.float64, device=DEVICE) if s.nx * s.ny <= 1 << 25 else None)
    torch.cuda.synchronize()  # the handle's stream does not wait for torch's
    return dict(kind="job", sim=sim, u0=u0, v0=v0, steps=case["steps"], out=out)


def run(state):
    if state["kind"] == "serve":
        server = state["server"]
        tickets = [server.submit(r) for r in state["requests"]]
        server.drain()
        return [list(server.result(t)[:3]) for t in tickets]
    sim, (u, v, P) = state["sim"], state["out"]
    sim.set_initial(state["u0"], state["v0"])
    sim.step(state["steps"])
    sim.fields_device(u, v, P)
    return [x for x in (u, v, P) if x is not None]


# ------------------------------------------------------------------ what a pass cannot do without
# floating-point operations of one node's iteration (moments and displacement
# update, gradient and stress, divergence, collision; no halo)
_FLOPS = {"nh": 155, "svk": 165, "le": 100}
# bytes of one node's state (nine populations and the displacement)
_STATE = {"fp64": 88, "fp32": 52, "fp16s": 34}
# a state beyond this many bytes cannot stay on the chip between iterations
_ON_CHIP = 129e6


def _lattice_work(nx, ny, steps, precision, model, inputs, outputs):
    n = nx * ny
    state = n * _STATE[precision]
    per_iteration = 2 * state if state > _ON_CHIP else 0
    return n * 8 * (inputs + outputs) + steps * per_iteration, n * steps * _FLOPS[model]


def work(case):
    if case["kind"] == "serve":
        w = [_lattice_work(r.nx, r.ny, r.nsteps, r.precision, r.model, 0, 8) for r in _requests(case, 0)]
    else:
        inputs = 2 if case["load"] == "periodic" else 4
        outputs = 8 if case["nx"] * case["ny"] <= 1 << 25 else 4
        w = [_lattice_work(case["nx"], case["ny"], case["steps"], case["precision"], case["model"], inputs, outputs)]
    return {"bytes": sum(b for b, _ in w), "flops": sum(f for _, f in w)}


# ------------------------------------------------------------------ the method in 64 bits
# Algorithm 1 of the paper with whole-lattice torch operations, one block
# after the other.
_EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
_EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
_OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
_W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
_LEFT, _RIGHT, _BOTTOM, _TOP = range(4)


def _load(e, k, dt, rho0):
    """Prescribed value of an edge at iteration k."""
    t = k * dt if e.unit == "time" else float(k)
    span = e.t1 - e.t0
    if e.shape == "const":
        f = 1.0
    elif e.shape in ("linear_ramp", "sin2_ramp"):
        f = min(max((t - e.t0) / span, 0.0), 1.0)
        f = f if e.shape == "linear_ramp" else math.sin(0.5 * math.pi * f) ** 2
    elif e.shape == "half_sine":
        f = math.sin(math.pi * (t - e.t0) / span) if e.t0 <= t < e.t1 else 0.0
    elif e.shape == "ricker":
        d = t - e.t0
        f = (1.0 - d * d / e.s) * math.exp(-0.5 * d * d / e.s) if t < e.t1 else 0.0
    else:  # disp_ramp
        f = rho0 / (span if e.unit == "time" else span * dt) if e.t0 <= t < e.t1 else 0.0
    return e.amp[0] * f, e.amp[1] * f


class _Reference:
    def __init__(self, s, u0, v0):
        self.s, self.h = s, s.spacing
        self.mu = s.E / (2 * (1 + s.nu))
        self.lam = s.E * s.nu / ((1 + s.nu) * (1 - 2 * s.nu))
        self.cs = math.sqrt(self.mu / s.rho0)
        self.c = math.sqrt(3) * self.cs
        self.dt = self.h / self.c
        self.per_x, self.per_y = s.edges[_LEFT].kind == "periodic", s.edges[_BOTTOM].kind == "periodic"
        zero = torch.zeros((2, s.ny, s.nx), dtype=torch.float64, device=DEVICE)
        self.u = zero.clone() if u0 is None else u0.permute(2, 0, 1).contiguous()
        v = zero if v0 is None else v0.permute(2, 0, 1)
        self.k = 0
        self.stress_and_source()
        H = self.gradient()
        self.f = self.equilibrium(-s.rho0 * (H[0] + H[3]), *(s.rho0 * v - 0.5 * self.dt * self.S),
                                  *self.flux(H)[[0, 1, 3]])

    def d(self, a, axis):
        """Finite difference: central, one-sided on a walled axis' ends."""
        if self.per_x if axis == 1 else self.per_y:
            return (torch.roll(a, -1, axis) - torch.roll(a, 1, axis)) / (2 * self.h)
        n, out = a.shape[axis], torch.empty_like(a)
        out.narrow(axis, 1, n - 2).copy_((a.narrow(axis, 2, n - 2) - a.narrow(axis, 0, n - 2)) / (2 * self.h))
        out.narrow(axis, 0, 1).copy_((a.narrow(axis, 1, 1) - a.narrow(axis, 0, 1)) / self.h)
        out.narrow(axis, n - 1, 1).copy_((a.narrow(axis, n - 1, 1) - a.narrow(axis, n - 2, 1)) / self.h)
        return out

    def gradient(self):
        return torch.stack([self.d(self.u[0], 1), self.d(self.u[0], 0), self.d(self.u[1], 1), self.d(self.u[1], 0)])

    def flux(self, H):
        tr = H[0] + H[3]
        o = -self.mu * (H[1] + H[2])
        return torch.stack([-self.mu * (2 * H[0] + tr), o, o, -self.mu * (2 * H[3] + tr)])

    def first_piola(self, H):
        mu, lam = self.mu, self.lam
        if self.s.model == "le":
            t, o = lam * (H[0] + H[3]), mu * (H[1] + H[2])
            return torch.stack([t + 2 * mu * H[0], o, o, t + 2 * mu * H[3]])
        F = (H[0] + 1, H[1], H[2], H[3] + 1)
        C = (F[0] * F[0] + F[2] * F[2], F[0] * F[1] + F[2] * F[3], F[1] * F[1] + F[3] * F[3])
        if self.s.model == "svk":
            e = (H[0] + 0.5 * (H[0] ** 2 + H[2] ** 2), 0.5 * (H[1] + H[2] + H[0] * H[1] + H[2] * H[3]),
                 H[3] + 0.5 * (H[1] ** 2 + H[3] ** 2))
            t = lam * (e[0] + e[2])
            S = (t + 2 * mu * e[0], 2 * mu * e[1], t + 2 * mu * e[2])
        else:
            J = F[0] * F[3] - F[1] * F[2]
            det = C[0] * C[2] - C[1] * C[1]
            inv = (C[2] / det, -C[1] / det, C[0] / det)
            t = 0.5 * lam * (J * J - 1)
            S = (t * inv[0] + mu * (1 - inv[0]), t * inv[1] - mu * inv[1], t * inv[2] + mu * (1 - inv[2]))
        return torch.stack([F[0] * S[0] + F[1] * S[1], F[0] * S[1] + F[1] * S[2],
                            F[2] * S[0] + F[3] * S[1], F[2] * S[1] + F[3] * S[2]])

    def stress_and_source(self):
        H, b = self.gradient(), self.s.body
        self.P = self.first_piola(H)
        self.N = self.P + self.flux(H)
        self.S = torch.stack([self.d(self.N[0], 1) + self.d(self.N[1], 0) + self.s.rho0 * b[0],
                              self.d(self.N[2], 1) + self.d(self.N[3], 0) + self.s.rho0 * b[1]])

    def equilibrium(self, r, jx, jy, pxx, pxy, pyy):
        cs2 = self.cs ** 2
        out = []
        for q in range(9):
            cx, cy = self.c * _EX[q], self.c * _EY[q]
            contr = ((pxx - r * cs2) * (cx * cx - cs2) + 2 * pxy * (cx * cy) + (pyy - r * cs2) * (cy * cy - cs2))
            out.append(_W[q] * (r + (cx * jx + cy * jy) / cs2 + contr / (2 * cs2 * cs2)))
        return torch.stack(out)

    def first(self, f):
        return (self.c * (f[1] - f[3] + f[5] - f[7] + f[8] - f[6]), self.c * (f[2] - f[4] + f[5] - f[7] + f[6] - f[8]))

    def step(self):
        s, c, dt = self.s, self.c, self.dt
        f = self.f
        r = f.sum(0)
        mx, my = self.first(f)
        jx, jy = mx + 0.5 * dt * self.S[0], my + 0.5 * dt * self.S[1]
        diag = f[5] + f[6] + f[7] + f[8]
        pi = (c * c * (f[1] + f[3] + diag), c * c * (f[5] - f[6] + f[7] - f[8]), c * c * (f[2] + f[4] + diag))
        g = f + (self.equilibrium(r, jx, jy, *pi) - f) / s.tau
        w = (1 - 0.5 / s.tau) * dt / self.cs ** 2
        for q in range(1, 9):
            g[q] += w * _W[q] * c * (_EX[q] * self.S[0] + _EY[q] * self.S[1])
        new = torch.stack([torch.roll(g[q], (_EY[q], _EX[q]), (0, 1)) for q in range(9)])
        self.walls(g, new, r, pi)
        mx, my = self.first(new)
        k = 0.5 * dt / s.rho0
        self.u[0] += k * (mx + 0.5 * dt * self.S[0] + jx)
        self.u[1] += k * (my + 0.5 * dt * self.S[1] + jy)
        self.f = new
        self.stress_and_source()
        self.k += 1

    def walls(self, g, new, r, pi):
        s = self.s
        if self.per_x and self.per_y:
            return
        load = [_load(e, self.k, self.dt, s.rho0) for e in s.edges]
        cs2 = self.cs ** 2
        for q in range(1, 9):
            ex, ey = _EX[q], _EY[q]
            wx = None if self.per_x or ex == 0 else (_RIGHT if ex > 0 else _LEFT)
            wy = None if self.per_y or ey == 0 else (_TOP if ey > 0 else _BOTTOM)
            col = s.nx - 1 if ex > 0 else 0
            row = s.ny - 1 if ey > 0 else 0
            # the nodes whose link q crosses the x wall only, the y wall only, both
            rows = slice(0, s.ny) if wy is None else (slice(0, s.ny - 1) if ey > 0 else slice(1, s.ny))
            cols = slice(0, s.nx) if wx is None else (slice(0, s.nx - 1) if ex > 0 else slice(1, s.nx))
            regions = []
            if wx is not None:
                regions.append((rows, slice(col, col + 1), wx, None))
            if wy is not None:
                regions.append((slice(row, row + 1), cols, None, wy))
            if wx is not None and wy is not None:
                regions.append((slice(row, row + 1), slice(col, col + 1), wx, wy))
            for ys, xs, ax, ay in regions:
                crossed = [w for w in (ax, ay) if w is not None]
                clamped = [w for w in crossed if s.edges[w].kind == "dirichlet"]
                out, c = g[q][ys, xs], self.c
                if clamped:
                    j = [sum(load[w][a] for w in clamped) / len(clamped) for a in range(2)]
                    out = out - 2 / cs2 * _W[q] * c * (ex * j[0] + ey * j[1])
                else:
                    at = lambda a: self.at_wall(a, ys, xs, ax, ay)  # noqa: E731
                    pxx, pxy, pyy = (at(p) for p in pi)
                    shear = []
                    if ax is not None:
                        n = 1.0 if ax == _RIGHT else -1.0
                        pxx = at(self.N[0]) - n * load[ax][0]
                        shear.append(at(self.N[2]) - n * load[ax][1])
                    if ay is not None:
                        n = 1.0 if ay == _TOP else -1.0
                        pyy = at(self.N[3]) - n * load[ay][1]
                        shear.append(at(self.N[1]) - n * load[ay][0])
                    pxy = sum(shear) / len(shear)
                    rw = at(r)
                    cx, cy = c * ex, c * ey
                    contr = ((pxx - rw * cs2) * (cx * cx - cs2) + 2 * pxy * (cx * cy)
                             + (pyy - rw * cs2) * (cy * cy - cs2))
                    out = -out + 2 * _W[q] * (rw + contr / (2 * cs2 * cs2))
                new[_OPP[q]][ys, xs] = out

    def at_wall(self, a, ys, xs, wx, wy):
        """A node field carried to the wall: the node's own value, or the
        two-point extrapolation across each crossed wall."""
        v = a[ys, xs]
        if self.s.extrap != "linear":
            return v
        e = v
        if wx is not None:
            i = 1 if wx == _LEFT else self.s.nx - 2
            e = e + 0.5 * (v - a[ys, i:i + 1])
        if wy is not None:
            i = 1 if wy == _BOTTOM else self.s.ny - 2
            e = e + 0.5 * (v - a[i:i + 1, xs])
        return e

    def fields(self):
        mx, my = self.first(self.f)
        v = torch.stack([mx + 0.5 * self.dt * self.S[0], my + 0.5 * self.dt * self.S[1]], -1) / self.s.rho0
        return self.u.permute(1, 2, 0).contiguous(), v, self.P.permute(1, 2, 0).contiguous()


def _exact_lattice(s, u0, v0, steps):
    ref = _Reference(s, u0, v0)
    for _ in range(steps):
        ref.step()
    return list(ref.fields())


def exact(case, seed):
    if case["kind"] == "serve":
        requests = _requests(case, seed)
        if sum(r.nsteps for r in requests) > 2600:
            return None
        return [[x.cpu().numpy() for x in _exact_lattice(r, None, None, r.nsteps)] for r in requests]
    if case["nx"] * case["ny"] > 1 << 25:
        return None  # minutes, and more memory than the card has
    s = _sim_case(case)
    return _exact_lattice(s, *_initial(case, s, seed), case["steps"])
