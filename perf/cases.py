"""What a program that uses this package has it do, as cases to time.

A case names a path (how the program drives the library), the data it runs on
and the sizes.  Every pass starts from the same inputs: it sets the state,
advances it and takes the result, as a program does with each new problem.

Paths:
  run        a fixed time step, Solver.run
  adaptive   the time step from the state's wave speed before every step
  logged     paper_2508_06273_gb300.runlog.run with a log line every step
  host       the state comes from and goes to pinned host memory every step
  batch      an ensemble of uneven grids, Batch.run
  fp64       the double-precision path of the accuracy studies
  surrogate  point values from the networks
  train      Adam steps of one network

Data: "vortex" (isentropic vortex at rest or moving), "smooth" (a few Fourier
modes), "riemann" (four constant states, run with every limiter and switch).
"""
import io
import math

import numpy as np
import torch

from paper_2508_06273_gb300 import af, runlog

GAMMA, CFL = 1.4, 0.3
PERIODIC, WALLS = "periodic", "walls"
BCS = {PERIODIC: (0, 0, 0, 0), WALLS: (1, 1, 2, 2), "outflow": (1, 1, 1, 1)}
# the option set of the four-quadrant problems
RIEMANN = {"tsw": 1, "limiter": 1, "flux_limiter": 1, "shock_blend": 1, "node_bounds": 1, "ubar": 1}
# the FP64 path takes no limiter
FP64 = {"limiter": 0, "fp64": 1}


def listed():
    return [
        # the smallest grid of the convergence tables and tests; launches and latency count
        {"name": "vortex_32", "path": "run", "data": "vortex", "speed": 1.0, "nx": 32, "ny": 32, "steps": 16},
        # a run with a log of its totals, minima and counters; outflow at the sides, walls
        # below and above, sizes that fill no tile
        {"name": "logged_walls_211x149", "path": "logged", "data": "smooth", "bc": WALLS, "nx": 211, "ny": 149, "steps": 8},
        # an ordinary grid of the convergence sweep, each time step from the wave speed
        {"name": "vortex_256", "path": "adaptive", "data": "vortex", "speed": 0.0, "nx": 256, "ny": 256, "steps": 8},
        # the two-stage linearisation of the tables, on a ragged grid
        {"name": "two_stage_389x301", "path": "run", "data": "smooth", "bc": PERIODIC, "lin_mode": 2, "nx": 389, "ny": 301, "steps": 6},
        # a large odd grid at a fixed step
        {"name": "vortex_1001x777", "path": "run", "data": "vortex", "speed": 0.0, "nx": 1001, "ny": 777, "steps": 6},
        # the benchmark's grid: a moving vortex on 8192^2
        {"name": "vortex_8192", "path": "adaptive", "data": "vortex", "speed": 1.0, "nx": 8192, "ny": 8192, "steps": 2},
        # Riemann data with every limiter and switch
        {"name": "riemann_600", "path": "adaptive", "data": "riemann", "nx": 600, "ny": 600, "steps": 4},
        # an ensemble of uneven grids, vortices and Riemann problems in turn, 64^2 to 512^2
        {"name": "ensemble_14", "path": "batch", "grids": 14, "lo": 64, "hi": 512, "steps": 10},
        # an accuracy study in double precision
        {"name": "fp64_192", "path": "fp64", "data": "vortex", "speed": 1.0, "nx": 192, "ny": 192, "steps": 4},
        # the learned point-value operator on smooth data
        {"name": "surrogate_640", "path": "surrogate", "data": "vortex", "speed": 0.0, "nx": 640, "ny": 640, "steps": 4},
        # training of one of its networks
        {"name": "train_4096", "path": "train", "rows": 200000, "batch": 4096, "steps": 24},
        # a program that moves the whole state through host memory every step
        {"name": "host_1024", "path": "host", "data": "vortex", "speed": 1.0, "nx": 1024, "ny": 1024, "steps": 2},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    path = rng.choice(["run", "run", "adaptive", "adaptive", "logged", "riemann", "batch", "fp64", "surrogate", "train", "host"])
    if path == "batch":
        lo = size(40, 90)
        return {"path": path, "grids": rng.randint(4, 15), "lo": lo, "hi": lo * rng.randint(2, 6), "steps": rng.randint(4, 12)}
    if path == "train":
        return {"path": path, "rows": size(20000, 400000), "batch": 8 * size(64, 2048), "steps": rng.randint(8, 32)}
    if path == "riemann":
        return {"path": "adaptive", "data": "riemann", "nx": size(40, 1200), "ny": size(40, 1200), "steps": rng.randint(2, 4)}
    if path == "surrogate":
        n = size(64, 1024)
        return {"path": path, "data": "vortex", "speed": 0.0, "nx": n, "ny": n, "steps": rng.randint(1, 5)}
    hi = {"run": 2600, "adaptive": 2600, "logged": 700, "fp64": 300, "host": 1500}[path]
    case = {"path": path, "nx": size(24, hi), "ny": size(24, hi), "steps": rng.randint(1, 3) if path == "host" else rng.randint(4, 9)}
    if path in ("fp64", "host") or rng.random() < 0.5:
        return dict(case, data="vortex", speed=rng.choice([0.0, 0.5, 1.0]))
    return dict(case, data="smooth", bc=rng.choice([PERIODIC, WALLS]), lin_mode=rng.choice([0, 0, 1, 2]))


# ------------------------------------------------------------------- inputs
def _vortex(rng, speed):
    """Centre and strength as in the seeded vortices of the convergence sweep,
    on the periodic box [0, 10]^2."""
    cx, cy = rng.uniform(3.0, 6.0, 2)
    eps = rng.uniform(3.0, 6.0)

    def f(x, y):
        X, Y = x - cx, y - cy
        X, Y = X - 10.0 * torch.floor(X / 10.0 + 0.5), Y - 10.0 * torch.floor(Y / 10.0 + 0.5)
        e = torch.exp(0.5 * (1.0 - X * X - Y * Y))
        T = 1.0 - (GAMMA - 1.0) * eps ** 2 / (8.0 * GAMMA * math.pi ** 2) * e * e
        rho = T ** (1.0 / (GAMMA - 1.0))
        w = eps / (2.0 * math.pi) * e
        return rho, speed - w * Y, speed + w * X, rho * T

    return f, 10.0, 10.0


def _smooth(rng, nx, ny):
    base = (1.0, 0.3, -0.2, 1.0)
    coef = rng.normal(size=(4, 3, 3, 2)) * 0.05
    lx, ly = 1.0, ny / nx

    def f(x, y):
        out = []
        for k in range(4):
            s = base[k] + 0.0 * (x + y)
            for a in range(3):
                for b in range(3):
                    ph = 2 * math.pi * (a * x / lx + b * y / ly)
                    s = s + coef[k, a, b, 0] * torch.cos(ph) + coef[k, a, b, 1] * torch.sin(ph)
            out.append(s)
        return out

    return f, lx, ly


def _riemann(rng, nx, ny):
    """Four states of the seeded four-quadrant problems, meeting at a point off
    the grid lines."""
    st = np.stack([rng.uniform(0.1, 1.5, 4), rng.uniform(-1.2, 1.2, 4), rng.uniform(-1.2, 1.2, 4), rng.uniform(0.01, 1.5, 4)], axis=1)
    lx, ly = 1.0, ny / nx
    xs = (int(nx * rng.uniform(0.4, 0.6)) + 0.5) / nx * lx
    ys = (int(ny * rng.uniform(0.4, 0.6)) + 0.5) / ny * ly

    def f(x, y):
        one = torch.ones_like(x + y)
        r, t = torch.heaviside(x - xs, 0.5 * torch.ones_like(x)), torch.heaviside(y - ys, 0.5 * torch.ones_like(y))
        w = ((1 - r) * (1 - t), r * (1 - t), (1 - r) * t, r * t)
        return [sum(float(st[q, k]) * w[q] for q in range(4)) * one for k in range(4)]

    return f, lx, ly


def _field(data, rng, nx, ny, speed=0.0):
    if data == "vortex":
        return _vortex(rng, speed)
    return _smooth(rng, nx, ny) if data == "smooth" else _riemann(rng, nx, ny)


def _discretise(f, lx, ly, nx, ny, periodic, dtype):
    """Cell averages (3 x 3 Gauss points) and point values on the GPU."""
    t = dict(dtype=torch.float64, device="cuda")
    dx, dy = lx / nx, ly / ny
    xn, yn = dx * torch.arange(nx + 1, **t), dy * torch.arange(ny + 1, **t)
    xc, yc = xn[:nx] + 0.5 * dx, yn[:ny] + 0.5 * dy

    def at(x, y):
        out = torch.empty((4, y.numel(), x.numel()), dtype=dtype, device="cuda")
        for j in range(0, y.numel(), 1024):
            for k, v in enumerate(f(x[None, :], y[j:j + 1024, None])):
                out[k, j:j + 1024] = v
        return out

    vtx, xe, ye = at(xn, yn), at(xn, yc), at(xc, yn)
    avg = torch.empty((4, ny, nx), dtype=dtype, device="cuda")
    g = math.sqrt(0.15)
    for j in range(0, ny, 1024):
        q = 0.0
        for a, wa in ((-g, 5 / 18), (0.0, 8 / 18), (g, 5 / 18)):
            for b, wb in ((-g, 5 / 18), (0.0, 8 / 18), (g, 5 / 18)):
                r, u, v, p = f((xc + a * dx)[None, :], (yc[j:j + 1024] + b * dy)[:, None])
                q = q + wa * wb * torch.stack([r, r * u, r * v, p / (GAMMA - 1.0) + 0.5 * r * (u * u + v * v)])
        avg[:, j:j + 1024] = q
    if periodic:
        vtx[:, :, nx], xe[:, :, nx] = vtx[:, :, 0], xe[:, :, 0]
        vtx[:, ny], ye[:, ny] = vtx[:, 0], ye[:, 0]
    return avg, vtx, xe, ye


def _speed(U):
    return (torch.maximum(U[1].abs(), U[2].abs()) + torch.sqrt(GAMMA * U[3] / U[0])).max()


def _prim(Q):
    u, v = Q[1] / Q[0], Q[2] / Q[0]
    return torch.stack([Q[0], u, v, (GAMMA - 1.0) * (Q[3] - 0.5 * Q[0] * (u * u + v * v))])


def _grid(case):
    bc = "outflow" if case["data"] == "riemann" else case.get("bc", PERIODIC)
    return case["nx"], case["ny"], bc


def _single(case, seed):
    """Sizes, boundary, spacings and input arrays of a single-grid case."""
    nx, ny, bc = _grid(case)
    f, lx, ly = _field(case["data"], np.random.default_rng(seed), nx, ny, case.get("speed", 0.0))
    dtype = torch.float64 if case["path"] == "fp64" else torch.float32
    return nx, ny, bc, lx / nx, ly / ny, _discretise(f, lx, ly, nx, ny, bc == PERIODIC, dtype)


def _fixed_dt(arrays, dx, dy):
    """The fixed time step of a run, with room for the wave speed to grow."""
    return 0.25 * min(dx, dy) / float(max(_speed(a) for a in (_prim(arrays[0]),) + arrays[1:]))


def _net(seed):
    """Parameters with the sizes of a trained network's: outputs of about 1e-3
    in the scaled units."""
    rng = np.random.default_rng(seed)
    p = [rng.normal(size=(128, 64)) / 8.0, 0.1 * rng.normal(size=128)]
    for _ in range(2):
        p += [rng.normal(size=(128, 128)) * math.sqrt(2.0 / 128), 0.1 * rng.normal(size=128)]
    w4 = np.zeros((16, 128))
    w4[:8] = rng.normal(size=(8, 128)) * 0.05
    p += [w4, np.zeros(16), np.full(64, 20.0), np.full(8, 1e-3)]
    net = af.Mlp(seed=1)
    net.set_params(np.concatenate([a.ravel() for a in p]).astype(np.float32))
    return net


def _batch_grids(case, seed):
    rng = np.random.default_rng(seed)
    for k in range(case["grids"]):
        # sizes belong to the case, data to the seed
        n = int(round(case["lo"] * (case["hi"] / case["lo"]) ** ((0.37 + 0.618034 * k) % 1.0)))
        data = "vortex" if k % 2 == 0 else "riemann"
        f, lx, ly = _field(data, rng, n, n, 1.0)
        yield n, data, f, lx, ly


def prepare(case, seed):
    path = case["path"]
    if path == "train":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        X = torch.randn((case["rows"], 64), device="cuda", generator=gen) * 0.05
        w = torch.randn((64, 8), device="cuda", generator=gen) * 0.1
        T = torch.tanh(X @ w) + 0.5 * (X @ w) ** 2
        net = af.Mlp(seed=5)
        net.fit_scales(X, T)
        return {"case": case, "net": net, "X": X, "T": T, "start": net.get_params(), "seed": seed % 1000 + 1}
    if path == "batch":
        grids = list(_batch_grids(case, seed))
        arrays = [_discretise(f, lx, ly, n, n, data == "vortex", torch.float32) for n, data, f, lx, ly in grids]
        b = af.Batch([(g[0], g[0]) for g in grids], [(g[3] / g[0], g[4] / g[0]) for g in grids],
                     bcs=[BCS[PERIODIC if g[1] == "vortex" else "outflow"] for g in grids])
        for k, g in enumerate(grids):
            for key, v in (RIEMANN if g[1] == "riemann" else {}).items():
                b.set_option(key, v, k)
        return {"case": case, "batch": b, "arrays": arrays}
    nx, ny, bc, dx, dy, arrays = _single(case, seed)
    options = RIEMANN if case["data"] == "riemann" else FP64 if path == "fp64" else {}
    s = af.Solver(nx, ny, dx, dy, GAMMA, BCS[bc], options=dict(options, lin_mode=case.get("lin_mode", 0)))
    state = {"case": case, "solver": s, "arrays": arrays, "h": min(dx, dy), "dt": _fixed_dt(arrays, dx, dy)}
    if path == "surrogate":
        s.set_surrogate(_net(seed + 1), _net(seed + 2))
    if path == "host":
        pinned = [a.cpu().pin_memory() for a in arrays]
        state |= {"pinned": pinned, "arrays": [a.numpy() for a in pinned]}
        state["out_t"] = [torch.empty_like(a).pin_memory() for a in pinned]
        state["out"] = [a.numpy() for a in state["out_t"]]
    return state


def run(state):
    case, steps = state["case"], state["case"]["steps"]
    path = case["path"]
    if path == "train":
        net = state["net"]
        net.set_params(state["start"])
        hist = net.train(state["X"], state["T"], steps, batch=case["batch"], lr=1e-3, seed=state["seed"])
        return {"loss": hist, "params": net.get_params()}
    if path == "batch":
        b = state["batch"]
        for k, a in enumerate(state["arrays"]):
            b.set_state(k, *a)
        b.set_end(math.inf, CFL)
        b.run(steps)
        return {"states": [b.get_state(k) for k in range(b.n)], "steps": b.query()[1]}
    s = state["solver"]
    if path == "host":
        for k in range(steps):
            s.set_state_host_async(*(state["arrays"] if k == 0 else state["out"]))
            s.step(CFL * state["h"] / s.max_speed())
            s.get_state_host_async(state["out"])
            s.host_sync()
        return dict(zip(("avg", "vtx", "xe", "ye"), state["out"]))
    if path == "fp64":
        s.set_state_f64(*state["arrays"])
        s.run(steps, state["dt"])
        return dict(zip(("avg", "vtx", "xe", "ye"), s.get_state_f64()))
    s.set_state(*state["arrays"])
    more = {}
    if path == "adaptive":
        for _ in range(steps):
            s.step(CFL * state["h"] / s.max_speed())
    elif path == "logged":
        log = io.StringIO()
        more["t"] = runlog.run(s, math.inf, CFL, state["h"], log=log, max_steps=steps)[0]
    else:
        s.run(steps, state["dt"])
    return dict(zip(("avg", "vtx", "xe", "ye"), s.get_state()), **more)


# --------------------------------------------------------------------- work
# A step of one cell: the state is 16 numbers (averages and three nodes of four
# variables) and the averages' low words, read and written; two levels of three
# nodes at about 450 operations of the bicharacteristic operator, the
# reconstruction, the correction term and the fluxes.
STEP_BYTES, STEP_FLOPS = 160.0, 3400.0
NET_FLOPS = 2.0 * (64 * 128 + 2 * 128 * 128 + 128 * 8)  # one row through the network


def work(case):
    path, steps = case["path"], case["steps"]
    if path == "train":
        rows = float(case["batch"]) * steps
        return {"bytes": rows * (64 + 8) * 4, "flops": 3 * rows * NET_FLOPS}
    if path == "batch":
        cells = float(sum(g[0] ** 2 for g in _batch_grids(case, 0)))
    else:
        cells = float(case["nx"] * case["ny"])
    size = 2.0 if path == "fp64" else 1.0
    step_bytes = {"fp64": 128.0}.get(path, STEP_BYTES) * size
    w = {"bytes": cells * (2 * 128.0 * size + steps * step_bytes), "flops": cells * steps * STEP_FLOPS}
    if path == "host":  # the state crosses the host link both ways every step
        w["bytes"] = cells * steps * (STEP_BYTES + 256.0)
    if path == "surrogate":
        w["flops"] = cells * steps * 3 * NET_FLOPS
    return w


# -------------------------------------------------------------------- exact
# The step in 64 bits with plain torch: the same method from its formulas, with
# the integrals over the Mach cone's base by Gauss quadrature on the arcs
# between the grid lines.
_GX, _GW = np.polynomial.legendre.leggauss(12)


def _axis(n, node, periodic, flip):
    """Sources and signs of the indices -2 .. n + 1 (+ 1 on grid lines)."""
    idx, sign = [], []
    last = n if node else n - 1
    for i in range(-2, last + 3):
        ghost = not periodic and (i < 0 or i > last)
        if periodic:
            idx.append(i % n)
        else:
            idx.append(i if not ghost else ((-i if node else -1 - i) if i < 0 else 2 * last - i + (0 if node else 1)))
        sign.append(-1.0 if ghost and flip else 1.0)
    t = dict(device="cuda")
    return torch.tensor(idx, **t), torch.tensor(sign, dtype=torch.float64, **t)


class _Exact:
    def __init__(self, nx, ny, bc, dx, dy, arrays, lin_mode):
        self.nx, self.ny, self.dx, self.dy, self.lin = nx, ny, dx, dy, lin_mode
        self.per, self.walls = bc == PERIODIC, bc == WALLS
        self.avg, self.n = arrays[0].double(), [a.double() for a in arrays[1:]]

    def state(self):
        return [self.avg] + self.n

    def speed(self):
        return float(max(_speed(a) for a in [_prim(self.avg)] + self.n))

    def pad(self, a, nodex, nodey):
        ix, sx = _axis(self.nx, nodex, self.per, False)
        iy, sy = _axis(self.ny, nodey, self.per, self.walls)
        a = a[:, iy][:, :, ix].clone()
        a[1] *= sx
        a[2] *= sy[:, None]
        return a

    def cells(self):
        """Monomials [a][b][var][cell] about the centre of the cells -1 .. n,
        and their primitive averages."""
        V, X, Y = self.pv, self.px, self.py
        nx, ny = self.nx, self.ny

        def c(a, di, dj):
            return a[:, 1 + dj:3 + dj + ny, 1 + di:3 + di + nx]

        f = [[c(V, 0, 0), c(X, 0, 0), c(V, 0, 1)], [c(Y, 0, 0), None, c(Y, 0, 1)], [c(V, 1, 0), c(X, 1, 0), c(V, 1, 1)]]
        Q = 36.0 * c(self.pad(self.avg, False, False), 0, 0)
        ub = 0.0
        for k in range(3):
            for l in range(3):
                if k == l == 1:
                    continue
                r, u, v, p = f[k][l]
                w = 4.0 if k == 1 or l == 1 else 1.0
                Q = Q - w * torch.stack([r, r * u, r * v, p / (GAMMA - 1.0) + 0.5 * r * (u * u + v * v)])
                ub = ub + w * f[k][l]
        f[1][1] = _prim(Q / 16.0)
        self.ub = (ub + 16.0 * f[1][1]) / 36.0
        r = [[f[1][l], f[2][l] - f[0][l], 2.0 * (f[0][l] + f[2][l]) - 4.0 * f[1][l]] for l in range(3)]
        self.m = torch.stack([torch.stack([r[1][a], r[2][a] - r[0][a], 2.0 * (r[0][a] + r[2][a]) - 4.0 * r[1][a]]) for a in range(3)])
        self.mf = self.m.reshape(3, 3, 4, -1)
        self.wc = nx + 2

    def poly(self, v, cell, x, y, more):
        m = self.mf[:, :, v][:, :, cell]
        if more:
            m = m[..., None]
        return sum(x ** a * y ** b * m[a, b] for a in range(3) for b in range(3))

    def eg2(self, kind, i, j, ul, tau):
        """EG2 at the nodes (i, j) of a kind (0 vertex, 1 x-edge, 2 y-edge),
        linearised about ul."""
        r0, u0, v0, p0 = ul
        c0 = torch.sqrt(GAMMA * p0 / r0)
        a, b = (u0 / c0).clamp(-1, 1), (v0 / c0).clamp(-1, 1)
        rx, ry, sx, sy = c0 * tau / self.dx, c0 * tau / self.dy, u0 * tau / self.dx, v0 * tau / self.dy
        cut = [q * 0.5 * math.pi + 0.0 * a for q in range(5)]
        if kind != 2:
            cut += [torch.acos(a), 2 * math.pi - torch.acos(a)]
        if kind != 1:
            cut += [torch.asin(b) % (2 * math.pi), math.pi - torch.asin(b)]
        cut = torch.stack(cut, 1).sort(1).values
        mid, half = 0.5 * (cut[:, 1:] + cut[:, :-1]), 0.5 * (cut[:, 1:] - cut[:, :-1])

        def local(X, Y):
            right = (X > 0).long() if kind != 2 else torch.zeros_like(X, dtype=torch.long)
            top = (Y > 0).long() if kind != 1 else torch.zeros_like(Y, dtype=torch.long)
            shape = [-1] + [1] * (X.dim() - 1)
            ci = i.view(shape) + (1 if kind == 2 else right)
            cj = j.view(shape) + (1 if kind == 1 else top)
            return cj * self.wc + ci, (0.0 if kind == 2 else 0.5 - right), (0.0 if kind == 1 else 0.5 - top)

        s = lambda q: q[:, None]  # noqa: E731
        cell, ox, oy = local(s(rx) * torch.cos(mid) - s(sx), s(ry) * torch.sin(mid) - s(sy))
        th = mid[..., None] + half[..., None] * torch.tensor(_GX, device="cuda")
        w = half[..., None] * torch.tensor(_GW, device="cuda")
        C, S = torch.cos(th), torch.sin(th)
        one = lambda q: q[..., None] if torch.is_tensor(q) else q  # noqa: E731
        X = rx[:, None, None] * C - sx[:, None, None] + one(ox)
        Y = ry[:, None, None] * S - sy[:, None, None] + one(oy)
        U, V, P = (self.poly(v, cell, X, Y, True) for v in (1, 2, 3))
        I = lambda q: (q * w).sum((1, 2)) / math.pi  # noqa: E731
        cell, ox, oy = local(-sx, -sy)
        rP, pP = self.poly(0, cell, ox - sx, oy - sy, False), self.poly(3, cell, ox - sx, oy - sy, False)
        z = I(P) - r0 * c0 * I(U * C + V * S)
        return torch.stack([rP - 2.0 * pP / c0 ** 2 + z / c0 ** 2,
                            I(-P * C / s(s(r0 * c0)) + U * (2 * C * C - 0.5) + 2 * V * S * C),
                            I(-P * S / s(s(r0 * c0)) + V * (2 * S * S - 0.5) + 2 * U * S * C), z - pP])

    def correction(self, kind, i, j, U):
        g = lambda a, di, dj: a[:, j + 2 + dj, i + 2 + di]  # noqa: E731
        cc = lambda di, dj: self.m[0, 0][:, j + 1 + dj, i + 1 + di]  # noqa: E731
        V, X, Y = self.pv, self.px, self.py
        if kind == 0:
            Ux, Uy = g(Y, 0, 0) - g(Y, -1, 0), g(X, 0, 0) - g(X, 0, -1)
        elif kind == 1:
            Ux, Uy = cc(0, 0) - cc(-1, 0), g(V, 0, 1) - g(V, 0, 0)
        else:
            Ux, Uy = g(V, 1, 0) - g(V, 0, 0), cc(0, 0) - cc(0, -1)
        (r, u, v, p), (rx, ux, vx, px), (ry, uy, vy, py) = U, Ux / self.dx, Uy / self.dy
        f1, f2 = ux * ux + uy * vx, uy * vx + vy * vy
        g1 = px * (GAMMA * (ux + vy) + ux) + py * vx
        g2 = py * (GAMMA * (ux + vy) + vy) + px * uy
        h1, h2 = (rx * px + ry * py) / r, (rx * u + ry * v) / r ** 2
        return torch.stack([r * (f1 + f2) + u * (rx * (2 * ux + vy) + ry * vx) + v * (rx * uy + ry * (ux + 2 * vy)) - h1,
                            u * f1 + v * uy * (ux + vy) + g1 / r - px * h2,
                            v * f2 + u * vx * (ux + vy) + g2 / r - py * h2,
                            u * g1 + v * g2 + GAMMA * p * (f1 + f2 - h1 / r)])

    def levels(self, kind, dt):
        """Point values of a kind at the half and the full step."""
        a = self.n[kind]
        ni, nj = a.shape[2], a.shape[1]
        new = [torch.empty_like(a), torch.empty_like(a)]
        flat = [q.view(4, -1) for q in new]
        for e in range(0, ni * nj, 120000):
            k = torch.arange(e, min(e + 120000, ni * nj), device="cuda")
            i, j = k % ni, k // ni
            U = a.reshape(4, -1)[:, k]
            ub = lambda di, dj: self.ub[:, j + 1 + dj, i + 1 + di]  # noqa: E731
            if self.lin == 1:
                ul = U
            elif self.lin == 2:
                ul = self.eg2(kind, i, j, U, 0.25 * dt)
            elif kind == 0:
                ul = 0.25 * (ub(0, 0) + ub(-1, 0) + ub(0, -1) + ub(-1, -1))
            else:
                ul = 0.5 * (ub(0, 0) + (ub(-1, 0) if kind == 1 else ub(0, -1)))
            if self.walls and kind != 1 and self.lin == 0:  # a wall's own nodes
                wall = (j == 0) | (j == self.ny)
                ul = torch.where(wall, U * torch.tensor([1.0, 1.0, 0.0, 1.0], device="cuda", dtype=torch.float64)[:, None], ul)
            T = self.correction(kind, i, j, U)
            for q, tau in enumerate((0.5 * dt, dt)):
                ul = self.eg2(kind, i, j, ul, tau) + 0.5 * tau * tau * T
                flat[q][:, k] = ul
        return new

    def step(self, dt):
        self.pv, self.px, self.py = self.pad(self.n[0], True, True), self.pad(self.n[1], True, False), self.pad(self.n[2], False, True)
        self.cells()
        lev = [self.levels(kind, dt) for kind in range(3)]

        def flux(kind, d):
            F = 0.0
            for U, w in ((self.n[kind], 1.0), (lev[kind][0], 4.0), (lev[kind][1], 1.0)):
                r, u, v, p = U
                un, E = (u, v)[d], p / (GAMMA - 1.0) + 0.5 * r * (u * u + v * v)
                F = F + w * torch.stack([r * un, r * u * un + (p if d == 0 else 0.0), r * v * un + (p if d == 1 else 0.0), un * (E + p)])
            return F

        V, W = flux(0, 0), flux(0, 1)
        Fx = (V[:, :-1] + 4.0 * flux(1, 0) + V[:, 1:]) / 36.0
        Gy = (W[:, :, :-1] + 4.0 * flux(2, 1) + W[:, :, 1:]) / 36.0
        self.avg = self.avg - dt / self.dx * (Fx[:, :, 1:] - Fx[:, :, :-1]) - dt / self.dy * (Gy[:, 1:] - Gy[:, :-1])
        self.n = [q[1] for q in lev]


def exact(case, seed):
    # The ensemble and the Riemann problems decide by comparisons which of
    # several updates a value takes, and the networks and their training run on
    # BF16 operands: a 64-bit evaluation is another computation there.
    if case["path"] in ("batch", "surrogate", "train") or case["data"] == "riemann":
        return None
    if case["nx"] * case["ny"] * case["steps"] > 6_000_000:  # too long
        return None
    nx, ny, bc, dx, dy, arrays = _single(case, seed)
    E = _Exact(nx, ny, bc, dx, dy, arrays, case.get("lin_mode", 0))
    fixed, t = _fixed_dt(arrays, dx, dy), 0.0
    for _ in range(case["steps"]):
        dt = fixed if case["path"] in ("run", "fp64") else CFL * min(dx, dy) / E.speed()
        E.step(dt)
        t += dt
    out = dict(zip(("avg", "vtx", "xe", "ye"), E.state()))
    return dict(out, t=t) if case["path"] == "logged" else out
