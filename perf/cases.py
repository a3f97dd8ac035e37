"""The solver's work as its users have it done: what is timed and compared when the code gets faster.

A pass is the run of an initial value problem: the initial state goes into a handle that the program keeps, the
scheme takes its time steps, and the final state (cell averages and face point values) comes back.  The drives:

* ``advance``  device state in, ``gks_advance`` (queued steps), device state out: how long runs are made
* ``step``     the same with one ``gks_step`` a step, its dt read on the host each time
* ``noalloc``  ``gks_step_noalloc``: one step between the caller's device arrays, no handle
* ``host``     page-locked host state in, one ``gks_step``, host state out: coupling with a host program each step
* ``batch``    independent grids of uneven sizes: host states in, ``gks_batch_step``, host averages out

The workloads are the paper's (Sections 4 and 5), in the sizes of the tests and the benchmark and around them.
FP32-bulk results are handed on in 32 bits, the precision of the scheme's fluxes and face values there.
"""
import math
import random
from types import SimpleNamespace

import numpy as np
import torch

from paper_1412_4489_gb300 import gks

PERIODIC, OUTFLOW, SLIP, ISOTHERMAL, ADIABATIC = range(5)
GAUSS = math.sqrt(3.0) / 6.0


def _case(name, family, drive, precision, nx, ny, steps, cfl=0.5, tau_eps=0.05, characteristic=0, grids=1, sizes=0):
    return {"name": name, "family": family, "drive": drive, "precision": precision, "nx": nx, "ny": ny, "steps": steps,
            "cfl": cfl, "tau_eps": tau_eps, "characteristic": characteristic, "grids": grids, "sizes": sizes}


def listed():
    return [
        # the smallest runs: a shock tube on one row of cells (Section 4.2); a step is all latency and launches
        _case("tube_200_fp64", "tube", "advance", "fp64", 200, 1, 60),
        # an accuracy study's mesh (Table 2: 81 x 81), stepped one call at a time at the paper's CFL number
        _case("vortex_81_fp64_steps", "vortex", "step", "fp64", 81, 81, 10, cfl=0.2, tau_eps=0.0),
        # a caller with its own memory management takes single FP64 steps of a small grid
        _case("riemann_96x80_fp64_noalloc", "riemann", "noalloc", "fp64", 96, 80, 1),
        # coupling with a host program: the state crosses the host link each way around one step
        _case("wave_384x256_fp64_host", "wave", "host", "fp64", 384, 256, 1, tau_eps=0.0),
        # walls, Navier-Stokes, strong gradients: the paper's viscous shock tube (300 x 150, Pr 0.73)
        _case("shock_tube_300x150_fp64", "viscous_tube", "advance", "fp64", 300, 150, 8),
        # the benchmark's grid in the precise form
        _case("wave_512_fp64", "wave", "advance", "fp64", 512, 512, 6, tau_eps=0.0),
        # the benchmark's headline: 512 x 512 smooth wave, FP32-bulk
        _case("wave_512_fp32", "wave", "advance", "fp32", 512, 512, 48, tau_eps=0.0),
        # viscous flow between a resting and a moving no-slip wall (Re 1000)
        _case("channel_512_fp32", "channel", "advance", "fp32", 512, 512, 24),
        # a ragged Navier-Stokes grid with discontinuities, reconstructed in characteristic variables
        _case("riemann_701x499_char_fp32", "riemann", "advance", "fp32", 701, 499, 10, characteristic=1),
        # four-quadrant Navier-Stokes data at the tests' full size
        _case("riemann_1024_fp32", "riemann", "advance", "fp32", 1024, 1024, 10),
        # the largest grid of the benchmark: far beyond the L2 cache
        _case("wave_4096_fp32", "wave", "advance", "fp32", 4096, 4096, 8, tau_eps=0.0),
        # many independent grids of uneven sizes in one launch
        _case("batch_48_fp32", "mixed", "batch", "fp32", 384, 384, 20, grids=48, sizes=5),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges.  FP64 grids up to 512^2 cells, FP32-bulk ones up to 4M; steps so that a pass
    stays below the largest listed one."""
    kind = rng.choice(["tube", "plane", "plane", "plane", "plane", "noalloc", "host", "batch"])
    precision = rng.choice(["fp32", "fp32", "fp64"])
    if kind == "tube":
        return _drawn("tube", "advance", precision, _log(rng, 50, 4000), 1, rng.randint(20, 40))
    if kind == "noalloc":
        nx, ny = _log(rng, 16, 256), _log(rng, 16, 256)
        family, te = rng.choice([("riemann", 0.05), ("wave", 0.0), ("channel", 0.05)])
        return _drawn(family, "noalloc", "fp64", nx, ny, 1, tau_eps=te)
    if kind == "host":
        return _drawn("wave", "host", "fp64", _log(rng, 48, 400), _log(rng, 48, 400), 1, tau_eps=0.0)
    if kind == "batch":
        steps = rng.randint(8, 20) if precision == "fp32" else rng.randint(2, 4)
        return _drawn("mixed", "batch", precision, 384, 384, steps, grids=rng.randint(8, 48 if precision == "fp32" else 12),
                      sizes=rng.randint(1, 1 << 20))
    family = rng.choice(["wave", "vortex", "riemann", "channel"] + (["viscous_tube"] if precision == "fp64" else []))
    if precision == "fp64":
        nx, ny = _log(rng, 24, 512), _log(rng, 24, 512)
        steps = rng.randint(2, 8)
    else:
        nx, ny = _log(rng, 32, 2048), _log(rng, 32, 2048)
        steps = max(4, min(10 if family == "riemann" else 24, (64 << 20) // (nx * ny)))
    return _drawn(family, rng.choice(["advance", "advance", "advance", "step"]), precision, nx, ny, steps,
                  cfl=0.2 if family == "vortex" else 0.5, tau_eps=0.0 if family in ("wave", "vortex") else 0.05,
                  characteristic=int(family in ("riemann", "viscous_tube") and rng.random() < 0.5))


def _drawn(*a, **kw):
    c = _case("", *a, **kw)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# initial states: cell averages and Gauss-point face values, made on the GPU
# ---------------------------------------------------------------------------
def _cons(rho, u, v, p, gamma):
    return torch.stack([rho, rho * u, rho * v, p / (gamma - 1.0) + 0.5 * rho * (u * u + v * v)])


def _grid(nx, ny, Lx, Ly, gamma, mu, Pr, bc):
    return SimpleNamespace(nx=nx, ny=ny, Lx=Lx, Ly=Ly, dx=Lx / nx, dy=Ly / ny, gamma=gamma, mu=mu, Pr=Pr, bc=bc)


def _points(g, dev):
    """Cell centres, and the Gauss points of the x- and y-faces: (x, y) pairs of broadcastable arrays."""
    ax = lambda n, h, o: (torch.arange(n, dtype=torch.float64, device=dev) + o) * h  # noqa: E731
    xc, yc = ax(g.nx, g.dx, 0.5)[None, :], ax(g.ny, g.dy, 0.5)[:, None]
    xf, yf = ax(g.nx + 1, g.dx, 0.0)[None, :], ax(g.ny + 1, g.dy, 0.0)[:, None]
    return (xc, yc), [(xf, yc + s * GAUSS * g.dy) for s in (-1, 1)], [(xc + s * GAUSS * g.dx, yf) for s in (-1, 1)]


def _fill_smooth(g, fn, dev):
    """Averages by a 3 x 3 Gauss-Legendre rule a cell, exact point values at the faces."""
    (xc, yc), px, py = _points(g, dev)
    z, w = [-math.sqrt(0.15), 0.0, math.sqrt(0.15)], [5 / 18, 8 / 18, 5 / 18]
    g.U = 0.0
    for a in range(3):
        for b in range(3):
            g.U = g.U + w[a] * w[b] * fn(xc + z[a] * g.dx, yc + z[b] * g.dy)
    g.U = g.U.contiguous()
    g.Wx = torch.stack([fn(x, y) for x, y in px], 1).contiguous()
    g.Wy = torch.stack([fn(x, y) for x, y in py], 1).contiguous()
    return g


def _fill_quadrants(g, states, xb, yb, width, dev):
    """Four states (north-east, north-west, south-west, south-east of (xb, yb)), the jumps between them spread over
    some cells: flow that the scheme has already worked on, whose rounding errors do not grow out of all bounds."""
    q = [_cons(*(torch.tensor(float(s), dtype=torch.float64, device=dev) for s in st), g.gamma) for st in states]

    def fn(x, y):
        x, y = torch.broadcast_tensors(x, y)
        e, n = 0.5 + 0.5 * torch.tanh((x - xb) / (width * g.dx)), 0.5 + 0.5 * torch.tanh((y - yb) / (width * g.dy))
        w = [e * n, (1 - e) * n, (1 - e) * (1 - n), e * (1 - n)]
        return sum(w[k][None] * q[k][:, None, None] for k in range(4))

    return _fill_smooth(g, fn, dev)


def _wave(nx, ny, r, dev, gamma=1.4, mu=0.0, Pr=1.0):
    phi = r.uniform(0.0, 2.0)

    def fn(x, y):
        rho = 1.0 + 0.2 * torch.sin(math.pi * (x + y) + phi)
        one = torch.ones_like(rho)
        return _cons(rho, one, one, one, gamma)

    return _fill_smooth(_grid(nx, ny, 2.0, 2.0, gamma, mu, Pr, [(PERIODIC, 0.0, 0.0, 1.0)] * 4), fn, dev)


def _vortex(nx, ny, r, dev):
    gamma, eps, x0, y0 = 1.4, r.uniform(4.0, 5.0), 5.0 + r.uniform(-0.5, 0.5), 5.0 + r.uniform(-0.5, 0.5)

    def fn(x, y):
        r2 = (x - x0) ** 2 + (y - y0) ** 2
        f = eps / (2 * math.pi) * torch.exp(0.5 * (1 - r2))
        T = 1 - (gamma - 1) * eps * eps / (8 * gamma * math.pi ** 2) * torch.exp(1 - r2)
        rho = T ** (1 / (gamma - 1))
        return _cons(rho, 1 - f * (y - y0), 1 + f * (x - x0), rho * T, gamma)

    return _fill_smooth(_grid(nx, ny, 10.0, 10.0, gamma, 0.0, 1.0, [(PERIODIC, 0.0, 0.0, 1.0)] * 4), fn, dev)


def _riemann(nx, ny, r, dev, gamma=1.4, mu=1e-4, Pr=0.72):
    states = [(r.uniform(0.3, 1.5), r.uniform(-0.6, 0.6), r.uniform(-0.6, 0.6), r.uniform(0.3, 1.5)) for _ in range(4)]
    return _fill_quadrants(_grid(nx, ny, 1.0, 1.0, gamma, mu, Pr, [(OUTFLOW, 0.0, 0.0, 1.0)] * 4), states, 0.5, 0.5, 8.0, dev)


def _tube(nx, r, dev):
    left = (r.uniform(0.9, 1.1), 0.0, 0.0, r.uniform(0.9, 1.1))
    right = (r.uniform(0.11, 0.14), 0.0, 0.0, r.uniform(0.09, 0.11))
    bc = [(OUTFLOW, 0.0, 0.0, 1.0)] * 2 + [(PERIODIC, 0.0, 0.0, 1.0)] * 2
    return _fill_quadrants(_grid(nx, 1, 1.0, 1.0 / nx, 1.4, 0.0, 1.0, bc), [right, left, left, right], 0.5, -100.0, 4.0, dev)


def _viscous_tube(nx, ny, r, dev):
    gamma, k = 1.4, r.uniform(0.9, 1.1)
    left, right = (120.0 * k, 0.0, 0.0, 120.0 * k / gamma), (1.2, 0.0, 0.0, 1.2 / gamma)
    wall = (ADIABATIC, 0.0, 0.0, 1.0)
    g = _grid(nx, ny, 1.0, 0.5, gamma, 1.0 / 200.0, 0.73, [wall, wall, wall, (SLIP, 0.0, 0.0, 1.0)])
    return _fill_quadrants(g, [right, left, left, right], 0.5, -100.0, 4.0, dev)


def _channel(nx, ny, r, dev):
    """Flow between a resting and a moving isothermal wall (Mach 0.1 to 0.2), periodic along them: the linear profile
    with a perturbation that vanishes at the walls."""
    gamma, lid, wave, p = 1.4, r.uniform(0.1, 0.2), r.uniform(0.02, 0.05), 1.0 / 1.4

    def fn(x, y):
        x, y = torch.broadcast_tensors(x, y)
        s = torch.sin(math.pi * y)
        u = lid * y + wave * torch.sin(2 * math.pi * x) * torch.sin(2 * math.pi * y)
        v = wave * torch.cos(2 * math.pi * x) * s * s
        one = torch.ones_like(u)
        return _cons(one, u, v, p * one, gamma)

    bc = [(PERIODIC, 0.0, 0.0, 1.0)] * 2 + [(ISOTHERMAL, 0.0, 0.0, p), (ISOTHERMAL, lid, 0.0, p)]
    return _fill_smooth(_grid(nx, ny, 1.0, 1.0, gamma, 0.15 / 1000.0, 0.72, bc), fn, dev)


def _sizes(case):
    """(nx, ny, gamma, mu) of each grid of a batch: sides 32..384, as in the benchmark's batch."""
    r = random.Random(case["sizes"])
    side = lambda: 32 * r.randint(1, max(1, case["nx"] // 32))  # noqa: E731
    return [(side(), side(), r.choice([1.4, 5.0 / 3.0]), 10.0 ** r.uniform(-4.0, -3.0)) for _ in range(case["grids"])]


def _initial(case, seed, dev):
    r = random.Random(seed * 7919 + 17)
    nx, ny, family = case["nx"], case["ny"], case["family"]
    if family == "mixed":
        return [(_wave if k % 2 == 0 else _riemann)(x, y, r, dev, gamma, mu, 0.72)
                for k, (x, y, gamma, mu) in enumerate(_sizes(case))]
    if family == "tube":
        return [_tube(nx, r, dev)]
    return [{"wave": _wave, "vortex": _vortex, "riemann": _riemann, "channel": _channel, "viscous_tube": _viscous_tube}[family](nx, ny, r, dev)]


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
class _State:
    """A handle (or batch), the states that go into it and the buffers that results come back in."""
    h = b = None

    def __del__(self):
        if self.h:
            gks.gks_destroy(self.h)
        if self.b:
            gks.gks_batch_destroy(self.b)


def _pinned(x):
    t = torch.empty(x.shape, dtype=torch.float64, pin_memory=True)
    t.copy_(x)
    return t


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    s = _State()
    s.case, s.stream = case, torch.cuda.Stream()
    precision = gks.GKS_FP32_BULK if case["precision"] == "fp32" else gks.GKS_FP64
    s.options = gks.gks_default_options(precision, tau_eps=case["tau_eps"], characteristic=case["characteristic"])
    grids = _initial(case, seed, dev)
    s.g = g = grids[0]
    if case["drive"] == "batch":
        s.grids = []
        for g in grids:
            host = [_pinned(x) for x in (g.U, g.Wx, g.Wy)]
            s.grids.append((host, [x.numpy() for x in host]))
        s.back = torch.empty(sum(4 * g.nx * g.ny for g in grids), dtype=torch.float64, pin_memory=True)
        s.out = torch.empty_like(s.back, dtype=torch.float32, pin_memory=True)
        s.b = gks.gks_batch_create(grids, s.options, s.stream.cuda_stream)
    elif case["drive"] == "host":
        s.host = [_pinned(x) for x in (g.U, g.Wx, g.Wy)]
        s.back = [torch.empty(x.shape, dtype=torch.float64, pin_memory=True) for x in s.host]
        s.h = gks.gks_create(g.nx, g.ny, g.Lx, g.Ly, g.gamma, g.Pr, g.mu, g.bc, s.options, s.stream.cuda_stream)
    else:
        s.back = [torch.empty_like(x) for x in (g.U, g.Wx, g.Wy)]
        if case["drive"] != "noalloc":
            s.h = gks.gks_create(g.nx, g.ny, g.Lx, g.Ly, g.gamma, g.Pr, g.mu, g.bc, s.options, s.stream.cuda_stream)
    torch.cuda.synchronize()
    return s


def _handed_on(s, values):
    """The results in the precision that they are used in."""
    if s.case["precision"] == "fp64":
        return values
    with torch.cuda.stream(s.stream):
        return [x.to(torch.float32) for x in values]


def run(s):
    c, g, drive, cfl = s.case, s.g, s.case["drive"], s.case["cfl"]
    if drive == "batch":
        for k, (_, (U, Wx, Wy)) in enumerate(s.grids):
            gks.gks_batch_set_state(s.b, k, U, Wx, Wy)
        gks.gks_batch_step(s.b, c["steps"], cfl)
        gks.gks_batch_sync(s.b)
        at, back, t = 0, s.back.numpy(), []
        for k, (_, (U, _, _)) in enumerate(s.grids):
            t.append(gks.gks_batch_get_state(s.b, k, back[at:at + U.size].reshape(U.shape))[0])
            at += U.size
        return {"U": s.out.copy_(s.back) if c["precision"] == "fp32" else s.back, "t": np.array(t)}
    if drive == "noalloc":
        dt = gks.gks_step_noalloc(g.nx, g.ny, g.Lx, g.Ly, g.gamma, g.Pr, g.mu, g.bc, s.options, g.U, g.Wx, g.Wy, *s.back,
                                  cfl, stream=s.stream.cuda_stream)
        return {"state": s.back, "t": dt}
    if drive == "host":
        gks.gks_set_state(s.h, *(x.numpy() for x in s.host))
        dt = gks.gks_step(s.h, cfl)
        gks.gks_get_state(s.h, *(x.numpy() for x in s.back))
        return {"state": s.back, "t": dt}
    gks.gks_set_state_device(s.h, g.U, g.Wx, g.Wy)
    if drive == "step":
        for _ in range(c["steps"]):
            gks.gks_step(s.h, cfl)
    else:
        gks.gks_advance(s.h, c["steps"], cfl)
    t = gks.gks_get_state_device(s.h, *s.back)
    return {"state": _handed_on(s, s.back), "t": t}


# operations of one face and one cell a step, counted on the scheme's formulas (an FMA is two)
FACE_EULER, FACE_NS, CELL = 1100, 1900, 500


def work(case):
    sizes = [(nx, ny, 1.0) for nx, ny, _, _ in _sizes(case)] if case["family"] == "mixed" else [
        (case["nx"], case["ny"], 1e-4 if case["family"] in ("riemann", "channel", "viscous_tube") else 0.0)]
    cells = sum(nx * ny for nx, ny, _ in sizes)
    faces = sum(nx * (ny + 1) + (nx + 1) * ny for nx, ny, _ in sizes)
    values = 4 * cells + 8 * faces
    out = (4 * cells if case["drive"] == "batch" else values) * (8 if case["precision"] == "fp64" else 4)
    flops = sum((nx * (ny + 1) + (nx + 1) * ny) * (FACE_NS if mu else FACE_EULER) + nx * ny * CELL for nx, ny, mu in sizes)
    return {"bytes": 8.0 * values + out, "flops": float(flops) * case["steps"]}


# ---------------------------------------------------------------------------
# the scheme in plain torch, 64 bits, term by term (arXiv:1412.4489)
# ---------------------------------------------------------------------------
CHUNK = 1 << 20  # faces that are evaluated together


def _half_moments(U, lam, n, kind):
    """<u^k>, k < n, of a unit Maxwellian over the whole line (0), u > 0 (1) or u < 0 (-1)."""
    if kind == 0:
        m = [torch.ones_like(U), U]
    else:
        edge = torch.exp(-lam * U * U) / (2 * torch.sqrt(math.pi * lam))
        h = 0.5 * torch.special.erfc(-kind * torch.sqrt(lam) * U)
        m = [h, U * h + kind * edge]
    for k in range(2, n):
        m.append(U * m[k - 1] + (k - 1) / (2 * lam) * m[k - 2])
    return m


class _Maxwellian:
    def __init__(self, w, K, kind=0):
        self.rho, self.U, self.V, self.K = w[0], w[1] / w[0], w[2] / w[0], K
        e = w[3] - 0.5 * (w[1] * self.U + w[2] * self.V)
        self.lam = (K + 2) * self.rho / (4 * e)
        self.p = self.rho / (2 * self.lam)
        self.mv, self.x2, self.x4 = _half_moments(self.V, self.lam, 7, 0), K / (2 * self.lam), K * (K + 2) / (4 * self.lam ** 2)
        self.over(kind)

    def over(self, kind):
        self.mu = _half_moments(self.U, self.lam, 8, kind)
        return self

    def mom(self, X, a, b):
        """<u^a v^b (X . psi) psi> / rho, psi = (1, u, v, (u^2 + v^2 + xi^2) / 2)."""
        z = lambda p, q: self.mu[a + p] * self.mv[b + q]  # noqa: E731
        z00, z10, z01, z20, z11, z02 = z(0, 0), z(1, 0), z(0, 1), z(2, 0), z(1, 1), z(0, 2)
        z22 = z(2, 2)
        e03 = 0.5 * (z20 + z02 + z00 * self.x2)
        e13 = 0.5 * (z(3, 0) + z(1, 2) + z10 * self.x2)
        e23 = 0.5 * (z(2, 1) + z(0, 3) + z01 * self.x2)
        e33 = 0.25 * (z(4, 0) + z(0, 4) + z00 * self.x4 + 2 * (z22 + (z20 + z02) * self.x2))
        rows = [(z00, z10, z01, e03), (z10, z20, z11, e13), (z01, z11, z02, e23), (e03, e13, e23, e33)]
        return torch.stack([r[0] * X[0] + r[1] * X[1] + r[2] * X[2] + r[3] * X[3] for r in rows])

    def unit(self, a):
        return torch.stack([self.mu[a], self.mu[a + 1], self.mu[a] * self.mv[1],
                            0.5 * (self.mu[a + 2] + self.mu[a] * (self.mv[2] + self.x2))])

    def solve(self, r):
        """X with <X . psi psi> / rho = r, over the whole velocity space."""
        U, V, lam, N = self.U, self.V, self.lam, self.K + 2
        q2 = U * U + V * V
        x4 = 4 * lam * lam / N * (2 * (r[3] - U * r[1] - V * r[2]) + (q2 - N / (2 * lam)) * r[0])
        x3 = 2 * lam * (r[2] - V * r[0]) - V * x4
        x2 = 2 * lam * (r[1] - U * r[0]) - U * x4
        return torch.stack([r[0] - U * x2 - V * x3 - x4 * (0.5 * q2 + N / (4 * lam)), x2, x3, x4])

    def coefficients(self, d):
        """The nine coefficients from the derivatives (n, t, nn, nt, tt) of the conservative variables."""
        kept, self.mu = self.mu, _half_moments(self.U, self.lam, 8, 0)
        c = SimpleNamespace()
        c.a1, c.a2, c.xx, c.xy, c.yy = (self.solve(d[k] / self.rho) for k in range(5))
        minus = lambda X, Y: self.solve(-(self.mom(X, 1, 0) + self.mom(Y, 0, 1)))  # noqa: E731
        c.A, c.tx, c.ty = minus(c.a1, c.a2), minus(c.xx, c.xy), minus(c.xy, c.yy)
        c.tt = minus(c.tx, c.ty)
        self.mu = kept
        return c

    def total(self, one, groups, a):
        """rho <u^a (one + sum of X u^p v^q) psi> over groups (X, p, q)."""
        return self.rho * (one * self.unit(a) + sum(self.mom(X, a + p, q) for X, p, q in groups))


def _time_weights(T, tau):
    """Integrals over [0, T] and values at T of C_1 .. C_8, C_7 t, C_7 t^2 (index 9, 10)."""
    x = torch.where(tau > 0, T / torch.where(tau > 0, tau, torch.ones_like(tau)), torch.full_like(tau, math.inf))
    e = torch.exp(-x)
    one = -torch.expm1(-x)
    xs = torch.clamp(x, max=1.0)
    s = [torch.zeros_like(x) for _ in range(6)]
    t = -xs
    for n in range(2, 26):
        t = t * (-xs / n)
        for k, w in enumerate((1, n - 1, n - 2, 0 if n < 3 else -1, -(n - 1) * (n - 4), 0 if n < 3 else -(n - 1) * (n - 2))):
            s[k] = s[k] + w * t
    small, t2, t3 = x < 1.0, tau * tau, tau ** 3
    pick = lambda a, b: torch.where(small, a, b)  # noqa: E731
    I, E = [None] * 11, [None] * 11
    I[1] = pick(tau * s[0], T - tau * one)
    I[2] = pick(t2 * s[2], 2 * t2 * one - tau * T * (1 + e))
    I[3] = pick(t2 * s[3], 0.5 * T * T - tau * T + t2 * one)
    I[4] = pick(-t3 * s[4], -4 * t3 + tau * (T + 2 * tau) ** 2 * e)
    I[9] = pick(t2 * s[1], t2 - tau * (tau + T) * e)
    I[10] = pick(t3 * s[5], 2 * t3 - tau * (T * T + 2 * T * tau + 2 * t2) * e)
    E[2] = pick(-tau * s[1], (T + tau) * e - tau)
    E[3] = pick(tau * s[0], T - tau + tau * e)
    I[5] = T ** 3 / 3 - tau * T * T
    I[6] = -tau * (0.5 * T * T + I[9])
    I[7], I[8] = tau * one, -I[9]
    E[1], E[4], E[5], E[6] = one, -(T * T + 2 * T * tau) * e, T * T - 2 * T * tau, -T * tau * (1 + e)
    E[7], E[8], E[9], E[10] = e, -T * e, T * e, T * T * e
    return I, E


def _evolve(L, R, avg, dn, dt, gamma, mu, Pr, T, tau_eps):
    """Time-integrated flux and the two Gauss-point values at T of faces: sides [6][4][F], averages [2][3][4][F]."""
    K = (4 - 2 * gamma) / (gamma - 1)
    sides = [_Maxwellian(L[0], K, 1), _Maxwellian(R[0], K, -1)]
    W0 = sum(m.rho * m.unit(0) for m in sides)
    g0 = _Maxwellian(W0, K)
    jump = torch.abs(sides[0].p - sides[1].p) / (sides[0].p + sides[1].p) * T
    ns = mu > 0
    tau = torch.where(ns, mu / g0.p + jump, tau_eps * T + jump)
    tn = torch.where(ns, tau, torch.zeros_like(tau))
    I, E = _time_weights(T, tau)
    y2 = dt * dt / 12
    (um, uc, up), (wm, wc, wp) = avg
    d = [((wp - up) + 2 * (wc - uc) + (wm - um)) / (4 * dn), (wp - wm + up - um) / (4 * dt),
         (26 * (wc + uc) - (wp + up + wm + um) - 48 * W0) / (8 * dn * dn), (wp - up - wm + um) / (2 * dn * dt),
         (wp - 2 * wc + wm + up - 2 * uc + um) / (2 * dt * dt)]
    c = g0.coefficients(d)

    def equilibrium(W):
        return W[1], [(W[3] * c.A + 0.5 * W[5] * c.tt + 0.5 * y2 * W[1] * c.yy, 0, 0), (W[2] * c.a1 + W[6] * c.tx, 1, 0),
                      (W[2] * c.a2 + W[6] * c.ty, 0, 1), (0.5 * W[4] * c.xx, 2, 0), (W[4] * c.xy, 1, 1), (0.5 * W[4] * c.yy, 0, 2)]

    F = g0.total(*equilibrium(I), 1)
    mean = g0.total(*equilibrium(I), 0)
    P0 = g0.total(*equilibrium(E), 0)
    zero = torch.zeros_like(T)
    P1 = g0.total(zero, [(E[1] * c.a2 + E[3] * c.ty, 0, 0), (E[2] * c.xy, 1, 0), (E[2] * c.yy, 0, 1)], 0)
    for m, S in zip(sides, (L, R)):
        k = m.coefficients(S[1:])

        def kinetic(W):
            return W[7], [(0.5 * y2 * W[7] * k.yy - tn * W[7] * k.A, 0, 0), ((W[8] - tn * W[7]) * k.a1 - tn * W[8] * k.tx, 1, 0),
                          ((W[8] - tn * W[7]) * k.a2 - tn * W[8] * k.ty, 0, 1), ((0.5 * W[10] - tn * W[8]) * k.xx, 2, 0),
                          ((W[10] - 2 * tn * W[8]) * k.xy, 1, 1), ((0.5 * W[10] - tn * W[8]) * k.yy, 0, 2)]

        F = F + m.total(*kinetic(I), 1)
        mean = mean + m.total(*kinetic(I), 0)
        P0 = P0 + m.total(*kinetic(E), 0)
        wy = -tn * E[7] - E[9]
        P1 = P1 + m.total(zero, [(E[7] * (k.a2 - tn * k.ty), 0, 0), (wy * k.xy, 1, 0), (wy * k.yy, 0, 1)], 0)
    u, v = g0.U, g0.V
    q2 = u * u + v * v
    q = F[3] - u * F[1] - v * F[2] + (0.5 * q2 + u * u) * F[0] - u * mean[3] + u * v * mean[2] - 0.5 * u * q2 * mean[0]
    F = torch.cat([F[:3], (F[3] + (1 / Pr - 1) * q)[None]])
    yg = GAUSS * dt
    return F, P0 - yg * P1, P0 + yg * P1


def _collisionless(a, b, gamma, T):
    """Flux and values of two constant states without collisions (the positivity fallback)."""
    K = (4 - 2 * gamma) / (gamma - 1)
    l, r = _Maxwellian(a, K, 1), _Maxwellian(b, K, -1)
    return T * (l.rho * l.unit(1) + r.rho * r.unit(1)), l.rho * l.unit(0) + r.rho * r.unit(0)


def _wall_average(kind, gamma, ut, Tw, w):
    """Boundary image of averages in the face frame (normal momentum first)."""
    if kind in (PERIODIC, OUTFLOW):
        return w
    r, n, t, e = w
    if kind == SLIP:
        return torch.stack([r, -n, t, e])
    if kind == ADIABATIC:
        return torch.stack([r, -n, 2 * r * ut - t, e + 2 * r * ut * ut - 2 * ut * t])
    return torch.stack([r, -n, 2 * r * ut - t, 2 * r * ut * ut - 2 * ut * t + (n * n + t * t) / r + 2 * r * Tw / (gamma - 1) - e])


def _wall_image(kind, gamma, ut, Tw, S):
    """Boundary image of a face state: value and (n, t, nn, nt, tt) derivatives mirrored in n."""
    if kind == OUTFLOW:
        return S
    sign = (1, -1, 1, 1, -1, 1)
    if kind in (SLIP, ADIABATIC):
        return torch.stack([sign[k] * _wall_average(kind, gamma, ut, Tw, S[k]) for k in range(6)])
    r, n, t, _ = S[0]
    m2, cT = n * n + t * t, 2 * Tw / (gamma - 1)

    def lin(a):
        return torch.stack([a[0], -a[1], 2 * ut * a[0] - a[2],
                            (2 * ut * ut - m2 / (r * r) + cT) * a[0] + 2 * n / r * a[1] + (2 * t / r - 2 * ut) * a[2] - a[3]])

    def hess(a, b):
        ma, mb = n * a[1] + t * a[2], n * b[1] + t * b[2]
        e = 2 * m2 / r ** 3 * a[0] * b[0] - 2 / (r * r) * (ma * b[0] + mb * a[0]) + 2 / r * (a[1] * b[1] + a[2] * b[2])
        z = torch.zeros_like(e)
        return torch.stack([z, z, z, e])

    return torch.stack([_wall_average(kind, gamma, ut, Tw, S[0]), -lin(S[1]), lin(S[2]), lin(S[3]) + hess(S[1], S[1]),
                        -(lin(S[4]) + hess(S[1], S[2])), lin(S[5]) + hess(S[2], S[2])])


def _swap(w, dim=0):
    return w.index_select(dim, torch.tensor([0, 2, 1, 3], device=w.device))


def _side(g, side):
    kind, u, v, Tw = g.bc[side]
    return kind, (v if side < 2 else u), Tw


def _padded(g, U):
    """Averages with the ghost ring; corners are x-images of y-ghosts."""
    per = g.bc[2][0] == PERIODIC
    img = lambda s, w: _swap(_wall_average(_side(g, s)[0], g.gamma, _side(g, s)[1], _side(g, s)[2], _swap(w)))  # noqa: E731
    U = torch.cat([img(2, U[:, -1:] if per else U[:, :1]), U, img(3, U[:, :1] if per else U[:, -1:])], 1)
    per = g.bc[0][0] == PERIODIC
    img = lambda s, w: _wall_average(_side(g, s)[0], g.gamma, _side(g, s)[1], _side(g, s)[2], w)  # noqa: E731
    return torch.cat([img(0, U[:, :, -1:] if per else U[:, :, :1]), U, img(1, U[:, :, :1] if per else U[:, :, -1:])], 2)


def _minmod(a, b):
    return torch.where(a * b > 0, torch.where(a.abs() < b.abs(), a, b), torch.zeros_like(a))


def _recon_scalar(st, dx, dy):
    """(a2, a3, a4, a5, a6) from the 13 stencil values (Section 3.2), weights with eps 1e-6 and C 10."""
    c, e, w, n, s, em, ep, wm, wp, nm, np_, sm, sp = st
    me, mw, mn, ms = (em + ep) / 2, (wm + wp) / 2, (nm + np_) / 2, (sm + sp) / 2
    a4 = _minmod(3 * (c + w - 2 * mw) / dx ** 2, 3 * (c + e - 2 * me) / dx ** 2)
    a2 = _minmod(2 * (c - mw) / dx + a4 * dx / 6, 2 * (me - c) / dx - a4 * dx / 6)
    a5 = _minmod(3 * (c + s - 2 * ms) / dy ** 2, 3 * (c + n - 2 * mn) / dy ** 2)
    a3 = _minmod(2 * (c - ms) / dy + a5 * dy / 6, 2 * (mn - c) / dy - a5 * dy / 6)
    r3 = math.sqrt(3.0) / (dx * dy)
    xe, xw = r3 * (ep - em) - a3 / dx, r3 * (wp - wm) - a3 / dx
    yn, ys = r3 * (np_ - nm) - a2 / dy, r3 * (sp - sm) - a2 / dy
    a6 = xe + yn
    for cand in (-xw + yn, -xw - ys, xe - ys):
        a6 = torch.where(cand.abs() < a6.abs() * (1 - 1e-8), cand, a6)
    c2, c4, c3, c5 = (e - w) / (2 * dx), (e - 2 * c + w) / dx ** 2, (n - s) / (2 * dy), (n - 2 * c + s) / dy ** 2
    c6 = r3 * ((ep - em) - (wp - wm) + (np_ - nm) - (sp - sm)) / 2
    I2 = (dx * c2) ** 2 + (dy * c3) ** 2 + 13 / 12 * ((dx * dx * c4) ** 2 + (dy * dy * c5) ** 2) + 7 / 6 * (dx * dy * c6) ** 2
    b1, b2 = (1e-6 + 10.0 * dx * dy) ** 2, (1e-6 + I2) ** 2
    w1 = b2 / (b1 + b2)
    return torch.stack([q + w1 * (p - q) for p, q in ((a2, c2), (a3, c3), (a4, c4), (a5, c5), (a6, c6))])


def _basis(w, gamma):
    """Left and right eigenvectors of the x-flux Jacobian: lists of rows, entries arrays."""
    rho = w[0]
    u, v = w[1] / rho, w[2] / rho
    q2 = u * u + v * v
    p = (gamma - 1) * (w[3] - 0.5 * rho * q2)
    c = torch.sqrt(gamma * p / rho)
    H, b1 = (w[3] + p) / rho, (gamma - 1) / (c * c)
    b2, o, z = 0.5 * b1 * q2, torch.ones_like(u), torch.zeros_like(u)
    R = [[o, o, z, o], [u - c, u, z, u + c], [v, v, o, v], [H - u * c, 0.5 * q2, v, H + u * c]]
    L = [[0.5 * (b2 + u / c), 0.5 * (-b1 * u - 1 / c), -0.5 * b1 * v, 0.5 * b1], [1 - b2, b1 * u, b1 * v, -b1], [-v, z, o, z],
         [0.5 * (b2 - u / c), 0.5 * (-b1 * u + 1 / c), -0.5 * b1 * v, 0.5 * b1]]
    return L, R


def _recon(g, P, Wx, Wy, characteristic):
    """Coefficients [5][4][ny][nx] of each cell's polynomial; cells not positive at a face centre get none."""
    dx, dy = g.dx, g.dy
    U = P[:, 1:-1, 1:-1]
    st = [U, P[:, 1:-1, 2:], P[:, 1:-1, :-2], P[:, 2:, 1:-1], P[:, :-2, 1:-1], Wx[:, 0, :, 1:], Wx[:, 1, :, 1:], Wx[:, 0, :, :-1],
          Wx[:, 1, :, :-1], Wy[:, 0, 1:], Wy[:, 1, 1:], Wy[:, 0, :-1], Wy[:, 1, :-1]]
    if not characteristic:
        a = _recon_scalar(st, dx, dy)
    else:
        mul = lambda M, w: torch.stack([sum(M[r][k] * w[k] for k in range(4)) for r in range(4)])  # noqa: E731
        L, R = _basis(U, g.gamma)
        x = [mul(R, m) for m in _recon_scalar([mul(L, w) for w in st], dx, dy)]
        L, R = _basis(_swap(U), g.gamma)
        y = [_swap(mul(R, m)) for m in _recon_scalar([mul(L, _swap(w)) for w in st], dx, dy)]
        a = torch.stack([x[0], y[1], x[2], y[3], 0.5 * (x[4] + y[4])])
    e0, n0 = U + a[2] * dx ** 2 / 12 - a[3] * dy ** 2 / 24, U + a[3] * dy ** 2 / 12 - a[2] * dx ** 2 / 24
    ok = torch.ones_like(U[0], dtype=torch.bool)
    for w in (e0 + a[0] * dx / 2, e0 - a[0] * dx / 2, n0 + a[1] * dy / 2, n0 - a[1] * dy / 2):
        ok = ok & (w[0] > 0) & (2 * w[0] * w[3] > w[1] ** 2 + w[2] ** 2)
    return torch.where(ok, a, torch.zeros_like(a))


def _axis_inputs(g, P, a, axis):
    """Sides, averages, and the constant states of every face of an axis, face frame, normal last: [.., t, n + 1]."""
    if axis == 1:  # transpose: x <-> y, momenta, coefficients
        P, a = _swap(P).transpose(1, 2), _swap(a, 1).index_select(0, torch.tensor([1, 0, 3, 2, 4], device=a.device)).transpose(2, 3)
    dn, dt = (g.dx, g.dy) if axis == 0 else (g.dy, g.dx)
    U = P[:, 1:-1, 1:-1]

    def state(s):
        sh = s * dn / 2
        return torch.stack([U + a[0] * sh + a[2] * dn ** 2 / 12 - a[3] * dt ** 2 / 24, a[0] + a[2] * sh, a[1] + a[4] * sh, a[2], a[4], a[3]])

    hi, lo = state(1), state(-1)
    s0, s1 = 2 * axis, 2 * axis + 1
    if g.bc[s0][0] == PERIODIC:
        first, last = hi[..., -1:], lo[..., :1]
    else:
        first = _wall_image(_side(g, s0)[0], g.gamma, _side(g, s0)[1], _side(g, s0)[2], lo[..., :1])
        last = _wall_image(_side(g, s1)[0], g.gamma, _side(g, s1)[1], _side(g, s1)[2], hi[..., -1:])
    avg = torch.stack([torch.stack([P[:, k:k + P.shape[1] - 2, m:m + P.shape[2] - 1] for k in range(3)]) for m in range(2)])
    return torch.cat([first, hi], -1), torch.cat([lo, last], -1), avg


def _wall_flux(g, axis, F):
    for side, at in ((2 * axis, 0), (2 * axis + 1, -1)):
        kind, ut, _ = _side(g, side)
        if kind in (SLIP, ISOTHERMAL, ADIABATIC):
            F[0, :, at] = 0.0
        if kind == ADIABATIC:
            F[3, :, at] = ut * F[2, :, at]
    return F


def _updated(g, F, U):
    (Fx, Fy) = F
    return U + (Fx[:, :, :-1] - Fx[:, :, 1:]) / g.dx + (Fy[:, :-1] - Fy[:, 1:]) / g.dy


def _not_physical(g, U):
    p = U[3] - 0.5 * (U[1] ** 2 + U[2] ** 2) / U[0]
    return ~((U[0] > 0) & (p > 0) & torch.isfinite(U).all(0))


def _rescued(g, P, U, F, W, new, dt):
    """The positivity fallback: collisionless fluxes at the faces of cells that are not physical, then everywhere."""
    T = torch.full((), dt, dtype=torch.float64, device=U.device)
    bad = _not_physical(g, new)
    for every in (False, True):
        if not bool(bad.any()):
            break
        for axis in range(2):
            Q = P if axis == 0 else _swap(P).transpose(1, 2)
            a, b = Q[:, 1:-1, :-1], Q[:, 1:-1, 1:]
            f, w = _collisionless(a, b, g.gamma, T)
            f = _wall_flux(g, axis, f.clone())
            m = bad if axis == 0 else bad.T
            per = g.bc[2 * axis][0] == PERIODIC
            pad = torch.cat([m[:, -1:] if per else torch.zeros_like(m[:, :1]), m, m[:, :1] if per else torch.zeros_like(m[:, :1])], 1)
            at = torch.ones_like(pad[:, 1:]) if every else pad[:, 1:] | pad[:, :-1]
            if axis == 1:
                f, w, at = _swap(f.transpose(1, 2)), _swap(w.transpose(1, 2)), at.T
            F[axis] = torch.where(at, f, F[axis])
            W[axis] = torch.where(at, w[:, None], W[axis])
        new = _updated(g, F, U)
        bad = _not_physical(g, new)
    return new


def _exact_step(grids, case, dev):
    inputs = []
    for g in grids:
        rho = g.U[0]
        u, v = g.U[1] / rho, g.U[2] / rho
        c = torch.sqrt(g.gamma * (g.gamma - 1) * (g.U[3] - 0.5 * rho * (u * u + v * v)) / rho)
        g.dt = case["cfl"] / float(torch.maximum((u.abs() + c) / g.dx, (v.abs() + c) / g.dy).max())
        g.P = _padded(g, g.U)
        a = _recon(g, g.P, g.Wx, g.Wy, case["characteristic"])
        for axis in range(2):
            inputs.append((g, axis, *_axis_inputs(g, g.P, a, axis)))
    flat = lambda k, lead: torch.cat([x[k].reshape(*lead, -1) for x in inputs], -1)  # noqa: E731
    each = lambda fn: torch.cat([torch.full((x[2][0, 0].numel(),), fn(x[0], x[1]), dtype=torch.float64, device=dev) for x in inputs])  # noqa: E731
    L, R, avg = flat(2, (6, 4)), flat(3, (6, 4)), flat(4, (2, 3, 4))
    con = [each(f) for f in (lambda g, x: g.dy if x else g.dx, lambda g, x: g.dx if x else g.dy, lambda g, x: g.gamma,
                             lambda g, x: g.mu, lambda g, x: g.Pr, lambda g, x: g.dt)]
    parts = [_evolve(L[..., k:k + CHUNK], R[..., k:k + CHUNK], avg[..., k:k + CHUNK], *(c[k:k + CHUNK] for c in con), case["tau_eps"])
             for k in range(0, L.shape[-1], CHUNK)]
    out, at = [torch.cat([p[k] for p in parts], -1) for k in range(3)], 0
    for k in range(0, len(inputs), 2):
        g, F, W = inputs[k][0], [None, None], [None, None]
        for axis in range(2):
            shape = inputs[k + axis][2].shape[2:]
            n = shape[0] * shape[1]
            f, wm, wp = (o[:, at:at + n].reshape(4, *shape) for o in out)
            at += n
            f, w = _wall_flux(g, axis, f.clone()), torch.stack([wm, wp], 1)
            F[axis], W[axis] = (f, w) if axis == 0 else (_swap(f.transpose(1, 2)), _swap(w.transpose(2, 3)))
        g.U = _rescued(g, g.P, g.U, F, W, _updated(g, F, g.U), g.dt)
        g.Wx, g.Wy, g.t = W[0], W[1], g.t + g.dt


def exact(case, seed, device=None):
    dev = torch.device(device or "cuda")
    grids = _initial(case, seed, dev)
    for g in grids:
        g.t = 0.0
    for _ in range(case["steps"]):
        _exact_step(grids, case, dev)
    if case["drive"] == "batch":
        return {"U": torch.cat([g.U.reshape(-1) for g in grids]), "t": np.array([g.t for g in grids])}
    g = grids[0]
    return {"state": [g.U.contiguous(), g.Wx.contiguous(), g.Wy.contiguous()], "t": g.t}
