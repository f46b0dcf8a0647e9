"""The work that users of this package run, as cases to be timed: one pass each.

A pass is what a program does between two looks at its simulation: put a state in (a checkpoint,
or the state another program hands over), advance it, take the state (and the fields) out; or the
gradient of an objective through a checkpointed rollout.  The flows, grids, orders, precisions and
parameters are those of ``paper_1910_13918_gb300/workloads.py`` and of the tests; the seed moves
the flow's phase, interface or vortex and adds the tests' 1e-4 noise.

``exact`` restates the method in FP64 with plain torch operations (per-axis Lagrange
interpolation, the equilibrium as a sum of products of per-axis Hermite moments) and shares no
code with the package.
"""
import itertools
import math

import torch

CV = 2.5            # gamma = 1.4
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f64": torch.float64}


def _case(name, kind, cells, order, prec="f32", steps=10, **more):
    axes = dict(zip(("cells_x", "cells_y", "cells_z"), cells))
    return dict(name=name, kind=kind, order=order, prec=prec, steps=steps, **axes, **more)


def listed():
    return [
        # the smallest configuration: 32 x 32 vertices, watched closely (fields and the mass and
        # energy sums every ten steps); nothing but latency
        _case("tgv_32_p2", "tgv", (16, 16), 2, ma=0.1, re=100.0, fields=True),
        # quasi-1D shock tube on a long strip with zero-gradient ends, state in L2
        _case("sod_8193x8_p2", "sod", (4096, 4), 2, steps=20),
        # the order 4 configuration, state larger than L2
        _case("tgv_1024_p4", "tgv", (256, 256), 4, steps=20, ma=0.3, re=1000.0),
        # a periodic grid of an odd number of vertices an axis: 341 cells of order 3
        _case("tgv_1023_p3", "tgv", (341, 341), 3, ma=0.3, re=1000.0),
        # the largest configuration: supersonic 2D Riemann problem, zero-gradient boundaries
        _case("riemann_3073_p3", "riemann", (1024, 1024), 3),
        # the same problem on 512 x 512 cells with BF16 storage
        _case("riemann_1537_p3_bf16", "riemann", (512, 512), 3, "bf16", steps=4),
        # the paper's 128 x 128-cell run of order 4 in FP64: the accuracy baseline
        _case("riemann_513_p4_f64", "riemann", (128, 128), 4, "f64", steps=4),
        # shock-vortex interaction on the transformed grid at Prandtl number 0.75
        _case("svi_1025x512_p2", "svi", (512, 256), 2, pr=0.75),
        # the D2Q9 comparison set: isothermal moving vortex
        _case("tgvm_2048_p4_d2q9", "tgvm", (512, 512), 4, velset="d2q9"),
        # 3D Taylor-Green vortex, D3Q125
        _case("tgv3d_128_p2", "tgv3d", (64, 64, 64), 2),
        # gradient of a weighted final density in the initial velocity: order 4 periodic grid, ...
        _case("grad_tgv_1024_p4", "tgv", (256, 256), 4, steps=10, ma=0.3, re=1000.0, grad=True, every=5),
        # ... and the shock-vortex interaction on a coarser transformed grid
        _case("grad_svi_257x128_p2", "svi", (128, 64), 2, steps=20, grad=True, every=10),
    ]


def draw(rng):
    def span(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    def cells(order, lo, hi):      # so that an axis has about lo to hi vertices
        return max(4, round(span(lo, hi) / order))

    pick = rng.choices(["tgv", "riemann", "sod", "svi", "tgvm", "tgv3d", "grad_tgv", "grad_svi"],
                       [4, 3, 1, 1, 2, 3, 2, 1])[0]
    order = rng.choice([1, 2, 3, 4])
    if pick in ("tgv", "riemann"):
        prec = rng.choices(["f32", "bf16", "f64"], [5, 2, 1])[0]
        top = 640 if prec == "f64" else 3072 if pick == "riemann" else 2048
        c = _case("", pick, (cells(order, 32, top), cells(order, 32, top)), order, prec,
                  4 if prec != "f32" else rng.choice([5, 10, 20]))
        if pick == "tgv":
            c.update(ma=rng.choice([0.1, 0.3]), re=rng.choice([100.0, 1000.0]), fields=rng.random() < 0.5)
    elif pick == "sod":
        c = _case("", "sod", (cells(order, 512, 16384), rng.randint(3, 12)), order, steps=20)
    elif pick == "svi":
        order = rng.choice([1, 2, 2, 3])
        ny = cells(order, 64, 512)
        c = _case("", "svi", (2 * ny + rng.randint(-3, 3), ny), order, rng.choice(["f32", "f32", "bf16"]), 4,
                  pr=rng.choice([1.0, 0.75]))
    elif pick == "tgvm":
        c = _case("", "tgvm", (cells(order, 32, 2048), cells(order, 32, 2048)), order,
                  rng.choice(["f32", "f32", "bf16"]), rng.choice([4, 10]),
                  velset=rng.choice(["d2q9", "d2q9", "d2q25"]))
    elif pick == "tgv3d":
        c = _case("", "tgv3d", tuple(cells(order, 16, 96) for _ in range(3)), order, "f32", rng.choice([2, 5]))
    elif pick == "grad_tgv":
        c = _case("", "tgv", (cells(order, 64, 1024), cells(order, 64, 1024)), order, steps=10, ma=0.3,
                  re=1000.0, grad=True, every=rng.choice([3, 5, 10]))
    else:
        ny = rng.randint(24, 64)
        c = _case("", "svi", (2 * ny, ny), 2, steps=10, grad=True, every=rng.choice([5, 10]))
    del c["name"]
    return c


# ---------------------------------------------------------------------------------------------
# grids, parameters and inputs of a case
# ---------------------------------------------------------------------------------------------
BOXES = {"tgv": ((0.0, 2 * math.pi),) * 2, "tgvm": ((0.0, 2 * math.pi),) * 2, "riemann": ((0.0, 1.0),) * 2,
         "svi": ((0.0, 2.0), (0.0, 1.0)), "tgv3d": ((0.0, 2 * math.pi),) * 3}
PERIODIC = {"tgv": (True, True), "tgvm": (True, True), "riemann": (False, False), "sod": (False, True),
            "svi": (False, True), "tgv3d": (True, True, True)}
SINE_MAP = 0.05     # amplitude of the transformed grid


class _Setup:
    """Grid, time step and relaxation time of a case, in plain numbers."""

    def __init__(self, case):
        self.kind, self.p, self.prec = case["kind"], case["order"], case["prec"]
        self.cells = [case[k] for k in ("cells_x", "cells_y", "cells_z") if k in case]
        self.dim = len(self.cells)
        self.box = BOXES.get(self.kind) or ((0.0, 1.0), (0.0, case["cells_y"] / case["cells_x"]))
        self.periodic = PERIODIC[self.kind]
        self.n = [c * self.p + (not per) for c, per in zip(self.cells, self.periodic)]
        self.mapped = self.kind == "svi"
        self.isothermal = self.kind == "tgvm"
        self.cv = 1.0 if self.isothermal else CV
        self.npop = 1 if self.isothermal else 2
        self.pr = case.get("pr", 1.0)
        if case.get("velset") == "d2q9":
            self.xi, self.w = [0.0, math.sqrt(3.0), -math.sqrt(3.0)], [2 / 3, 1 / 6, 1 / 6]
        else:
            s10 = math.sqrt(10.0)
            s, l = math.sqrt(5.0 - s10), math.sqrt(5.0 + s10)
            self.xi = [0.0, s, l, -s, -l]
            self.w = [8 / 15] + [(7 + 2 * s10) / 60, (7 - 2 * s10) / 60] * 2
        self.q = len(self.xi) ** self.dim
        h = min((hi - lo) / (c * self.p) for (lo, hi), c in zip(self.box, self.cells))
        self.dt = 0.5 * h / (math.sqrt(5.0 + math.sqrt(10.0)) * math.sqrt(self.dim))   # CFL 0.5
        if self.kind == "sod":
            self.tau = 1.518
        elif self.kind == "svi":   # the departures reach 4.4 vertex spacings
            self.dt, self.tau = 1.536 * h, 0.8333
        elif self.kind == "riemann":
            self.tau = 1.94815
        else:
            nu = {"tgv": lambda: case["ma"] * 2 * math.pi / case["re"],
                  "tgvm": lambda: 0.01 * 2 * math.pi / 10.0, "tgv3d": lambda: 0.1 / 1600.0}[self.kind]()
            self.tau = nu / self.dt + 0.5
        self.nv = math.prod(self.n)

    def nodes(self):               # Gauss-Lobatto-Chebyshev points of the unit cell
        return [0.5 * (1.0 - math.cos(k * math.pi / self.p)) for k in range(self.p + 1)]

    def axis(self, d, device):     # reference coordinates of the vertices of one axis
        (lo, hi), c = self.box[d], self.cells[d]
        j = torch.arange(self.n[d], device=device)
        nodes = torch.tensor(self.nodes()[:-1], dtype=torch.float64, device=device)
        return lo + (hi - lo) / c * (torch.div(j, self.p, rounding_mode="floor") + nodes[j % self.p])

    def coords(self, device):      # physical coordinates, arrays of shape (.., ny, nx)
        ref = torch.meshgrid(*[self.axis(d, device) for d in reversed(range(self.dim))], indexing="ij")[::-1]
        return _sine_map(*ref) if self.mapped else ref

    def velocities(self):          # component indices per velocity, the last one fastest
        return list(itertools.product(range(len(self.xi)), repeat=self.dim))


def _sine_map(xi, eta):
    a, pi = SINE_MAP, math.pi
    return (xi + a * torch.sin(2 * pi * xi) * torch.sin(pi * eta),
            eta + a * torch.sin(pi * xi) * torch.sin(2 * pi * eta))


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _flow(case, seed):
    """Initial (rho, u, T) of the case, FP64: u a list of the velocity components."""
    s, device = _Setup(case), _device()
    gen = torch.Generator(device=device).manual_seed(int(seed))
    a, b, c = torch.rand(3, generator=gen, device=device, dtype=torch.float64).tolist()
    x, y, *z = s.coords(device)
    if s.kind == "tgv":
        x, y, ma = x + 2 * math.pi * a, y + 2 * math.pi * b, case["ma"] * (0.9 + 0.2 * c)
        rho, u = torch.ones_like(x), [ma * torch.sin(x) * torch.cos(y), -ma * torch.cos(x) * torch.sin(y)]
        T = 1.0 + ma * ma / 4 * (torch.cos(2 * x) + torch.cos(2 * y))
    elif s.kind == "tgvm":
        x, y, uv, uh = x + 2 * math.pi * a, y + 2 * math.pi * b, 0.01, 0.05 * c
        rho = 1.0 + uv * uv / 4 * (torch.cos(2 * x) + torch.cos(2 * y))
        u = [uh + uv * torch.sin(x) * torch.cos(y), -uv * torch.cos(x) * torch.sin(y)]
        T = torch.ones_like(x)
    elif s.kind == "sod":
        left = x < 0.45 + 0.1 * a
        rho = torch.where(left, 1.0, 0.125).double()
        u, T = [torch.zeros_like(x), torch.zeros_like(x)], torch.where(left, 1.0, 0.8).double()
    elif s.kind == "riemann":      # the states of the paper's Table III
        east, north = x >= 0.45 + 0.1 * a, y >= 0.45 + 0.1 * b

        def quadrants(ne, nw, sw, se):
            return torch.where(north, torch.where(east, ne, nw), torch.where(east, se, sw)).double()

        rho = quadrants(0.5313, 1.0, 0.8, 1.0)
        u = [quadrants(0.0, 0.7276, 0.0, 0.0), quadrants(0.0, 0.0, 0.0, 0.7276)]
        T = quadrants(0.4, 1.0, 1.0, 1.0) / rho
    elif s.kind == "svi":          # stationary Mach 1.2 shock, isentropic vortex ahead of it
        g, ma, mv, radius = 1.4, 1.2, 0.25, 0.075
        m2 = ma * ma
        rr, pp = (g + 1) * m2 / ((g - 1) * m2 + 2), 1 + 2 * g / (g + 1) * (m2 - 1)
        ahead, dx, dy = x < 0.5, x - 0.2 - 0.1 * a, y - 0.4 - 0.2 * b
        r2 = (dx * dx + dy * dy) / radius ** 2
        env, base = torch.exp(0.5 * (1 - r2)), 1 - 0.5 * (g - 1) * mv * mv * torch.exp(1 - r2)
        rho = torch.where(ahead, base ** (1 / (g - 1)), rr)
        u = [torch.where(ahead, ma - mv * env * dy / radius, ma / rr),
             torch.where(ahead, mv * env * dx / radius, 0.0)]
        T = torch.where(ahead, base ** (g / (g - 1)), pp) / g / rho
    else:                          # 3D Taylor-Green vortex
        x, y, z, ma = x + 2 * math.pi * a, y + 2 * math.pi * b, z[0] + 2 * math.pi * c, 0.1
        rho = torch.ones_like(x)
        u = [ma * torch.sin(x) * torch.cos(y) * torch.cos(z), -ma * torch.cos(x) * torch.sin(y) * torch.cos(z),
             torch.zeros_like(x)]
        T = 1.0 + ma * ma / 16 * (torch.cos(2 * x) + torch.cos(2 * y)) * (torch.cos(2 * z) + 2.0)

    def noise():
        return 1e-4 * torch.randn(x.shape, generator=gen, device=device, dtype=torch.float64)

    speed = max(max(float(v.abs().max()) for v in u), 1e-3)
    rho, u = rho * (1 + noise()), [v + speed * noise() for v in u]
    return rho, u, T if s.isothermal else T * (1 + noise())


def _equilibrium(s, rho, u, T):
    """f^eq (and g^eq = (2 C_v - D) T f^eq), one velocity plane at a time: full populations."""
    q = torch.zeros_like(T) if s.isothermal else T - 1.0
    A = [[torch.ones_like(v), v, v * v + q, v ** 3 + 3 * v * q, v ** 4 + 6 * v * v * q + 3 * q * q] for v in u]
    he = [[1.0, x, (x * x - 1) / 2, (x ** 3 - 3 * x) / 6, (x ** 4 - 6 * x * x + 3) / 24] for x in s.xi]
    X = [[[A[d][k] * he[a][k] for k in range(5)] for a in range(len(s.xi))] for d in range(s.dim)]
    for comps in s.velocities():
        total = [X[0][comps[0]][k] for k in range(5)]      # [m]: terms of order m over the axes so far
        for d in range(1, s.dim):
            total = [sum(total[j] * X[d][comps[d]][m - j] for j in range(m + 1)) for m in range(5)]
        f = math.prod(s.w[c] for c in comps) * rho * sum(total)
        yield torch.stack([f, (2 * s.cv - s.dim) * T * f]) if s.npop == 2 else f[None]


def _weights(s):
    """Lattice weights of the populations, [npop][q]."""
    w = [math.prod(s.w[c] for c in comps) for comps in s.velocities()]
    return [w, [(2 * s.cv - s.dim) * x for x in w]][: s.npop]


def _state(case, seed):
    """The state a pass starts from, as the package exchanges it: deviations from the lattice
    weights in the storage type in 2D, full FP64 populations in FP64 and in 3D."""
    s = _Setup(case)
    full = s.prec == "f64" or s.dim == 3
    flow = _flow(case, seed)
    out = torch.empty([s.npop, s.q] + s.n[::-1], dtype=torch.float64 if full else DTYPES[s.prec],
                      device=flow[0].device)
    w = _weights(s)
    for i, f in enumerate(_equilibrium(s, *flow)):
        for k in range(s.npop):
            out[k, i] = f[k] if full else f[k] - w[k][i]
    return out


def _objective(case, seed):
    """Weights of the final density in the objective: a smooth positive sensor field."""
    s, device = _Setup(case), _device()
    x, y = s.coords(device)
    k = 1 + int(seed) % 3
    (x0, x1), (y0, y1) = s.box
    return (1.5 + torch.sin(2 * math.pi * k * (x - x0) / (x1 - x0)) * torch.cos(2 * math.pi * (y - y0) / (y1 - y0))) / s.nv


# ---------------------------------------------------------------------------------------------
# the passes
# ---------------------------------------------------------------------------------------------
_STREAM = []


def _stream():
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


def prepare(case, seed):
    from paper_1910_13918_gb300.sllbm import SLLBM, SLLBM3D
    s = _Setup(case)
    bc = [0 if per else 1 for per in s.periodic]
    with torch.cuda.stream(_stream()):
        if s.dim == 3:
            sim = SLLBM3D(cells=tuple(s.cells), order=s.p, box=s.box, bc=tuple(bc), dt=s.dt, tau=s.tau, cv=s.cv,
                          prec=s.prec, stream=_stream())
        else:
            (x0, x1), (y0, y1) = s.box
            sim = SLLBM(nx_cells=s.cells[0], ny_cells=s.cells[1], order=s.p, x0=x0, x1=x1, y0=y0, y1=y1,
                        bc_x=bc[0], bc_y=bc[1], dt=s.dt, tau=s.tau, cv=s.cv, prec=s.prec,
                        map_kind=1 if s.mapped else 0, map_a=SINE_MAP if s.mapped else 0.0, pr=s.pr,
                        isothermal=s.isothermal, velset=case.get("velset", "d2q25"), stream=_stream())
        sim.precompute()
        state = {"case": case, "sim": sim}
        if case.get("grad"):
            rho, (u, v), T = _flow(case, seed)
            state.update(rho=rho, T=T, u=u.requires_grad_(), v=v.requires_grad_(), weight=_objective(case, seed))
        else:
            state["in"] = _state(case, seed)
            if s.dim == 2:
                state["out"] = torch.empty_like(state["in"])
    torch.cuda.synchronize()
    return state


def run(state):
    case, sim = state["case"], state["sim"]
    with torch.cuda.stream(_stream()):
        # 3D states and rollout fields come widened to FP64 from FP32 arithmetic; a program that
        # runs in FP32 keeps them as FP32
        if case.get("grad"):
            from paper_1910_13918_gb300.autograd import rollout
            rho = rollout(sim, state["u"], state["v"], state["rho"], state["T"], case["steps"], case["every"])
            du, dv = torch.autograd.grad(rho, (state["u"], state["v"]), state["weight"])
            return {"rho": rho.detach().float(), "du": du.float(), "dv": dv.float()}
        sim.set_state(state["in"])
        sim.step(case["steps"])
        if "cells_z" in case:
            return {"state": sim.get_state().float()}
        out = {}
        if case.get("fields"):
            m = sim.moments()
            out = {k: m[k] for k in ("rho", "u", "v", "T")}
            out["sums"] = torch.tensor([m["mass"], m["energy"]], dtype=torch.float32)
        out["state"] = sim.get_state(out=state["out"])
        return out


def work(case):
    """A step reads every population once and writes it once, in its storage type; an adjoint step
    the FP32 adjoint populations and four moments a vertex."""
    s = _Setup(case)
    updates = s.nv * s.q * s.npop * case["steps"]
    elem = {"f32": 4, "bf16": 2, "f64": 8}[s.prec]
    per = 2 * s.dim * (s.p + 1) + 16
    if case.get("grad"):           # forward, recomputation from the checkpoints, adjoint
        return {"bytes": 2 * updates * 2 * elem + case["steps"] * s.nv * 416, "flops": 3 * updates * per}
    return {"bytes": updates * 2 * elem, "flops": updates * per}


# ---------------------------------------------------------------------------------------------
# the same passes in FP64 with plain torch
# ---------------------------------------------------------------------------------------------
def _fold(x, box, periodic):
    lo, hi = box
    return lo + torch.remainder(x - lo, hi - lo) if periodic else x.clamp(lo, hi)


def _stencil(s, d, x):
    """Stencil indices and Lagrange weights, [p + 1] tensors of x's shape, at reference points x."""
    (lo, hi), c = s.box[d], s.cells[d]
    t = (x - lo) / ((hi - lo) / c)
    cell = t.floor().clamp(0, c - 1)
    r, nodes = t - cell, s.nodes()
    idx = [(cell.long() * s.p + k) % s.n[d] for k in range(s.p + 1)]
    return idx, [math.prod((r - m) / (nodes[k] - m) for j, m in enumerate(nodes) if j != k) for k in range(s.p + 1)]


def _departures(s, device):
    """Per velocity, a function that interpolates a plane [npop][..][ny][nx] at its departures."""
    if s.mapped:
        X, Y = s.coords(device)
        out = []
        for a, b in s.velocities():
            x = _fold(X - s.dt * s.xi[a], s.box[0], s.periodic[0])
            y = _fold(Y - s.dt * s.xi[b], s.box[1], s.periodic[1])
            xi, eta, m, pi = x.clone(), y.clone(), SINE_MAP, math.pi
            for _ in range(12):    # Newton inversion of the map
                fx, fy = _sine_map(xi, eta)
                fx, fy = fx - x, fy - y
                j11 = 1 + 2 * pi * m * torch.cos(2 * pi * xi) * torch.sin(pi * eta)
                j12 = pi * m * torch.sin(2 * pi * xi) * torch.cos(pi * eta)
                j21 = pi * m * torch.cos(pi * xi) * torch.sin(2 * pi * eta)
                j22 = 1 + 2 * pi * m * torch.sin(pi * xi) * torch.cos(2 * pi * eta)
                det = j11 * j22 - j12 * j21
                xi, eta = xi - (j22 * fx - j12 * fy) / det, eta - (j11 * fy - j21 * fx) / det
            (ix, wx), (iy, wy) = _stencil(s, 0, xi.clamp(*s.box[0])), _stencil(s, 1, eta.clamp(*s.box[1]))
            terms = [((iy[l] * s.n[0] + ix[k]).reshape(-1), (wy[l] * wx[k]).reshape(-1))
                     for l in range(s.p + 1) for k in range(s.p + 1)]
            out.append(lambda F, terms=terms: sum(F.flatten(1)[:, i] * w for i, w in terms).reshape(F.shape))
        return out
    tables = [[_stencil(s, d, _fold(s.axis(d, device) - s.dt * x, s.box[d], s.periodic[d])) for x in s.xi]
              for d in range(s.dim)]

    def along(F, d, comp):
        idx, w = tables[d][comp]
        shape = [-1] + [1] * d
        return sum(F.index_select(F.dim() - 1 - d, i) * v.reshape(shape) for i, v in zip(idx, w))

    def at(comps):
        def interpolate(F):
            for d, c in enumerate(comps):
                F = along(F, d, c)
            return F
        return interpolate
    return [at(comps) for comps in s.velocities()]


def _moments(s, F):
    comps = s.velocities()
    rho = sum(F[0, i] for i in range(s.q))
    u = [sum(F[0, i] * s.xi[c[d]] for i, c in enumerate(comps)) / rho for d in range(s.dim)]
    e = sum(F[0, i] * sum(s.xi[k] ** 2 for k in c) for i, c in enumerate(comps))
    if s.npop == 2:
        e = e + sum(F[1, i] for i in range(s.q))
    return rho, u, (e - rho * sum(v * v for v in u)) / (2 * s.cv * rho)


def _collide(s, F):
    """Post-collision populations; F is a tensor [npop][q][..]."""
    rho, u, T = _moments(s, F)
    omega, planes = 1.0 / s.tau, []
    extra = None
    if s.pr != 1.0:                # quasi-equilibrium of the centred third moments
        powers = [(3, 0), (2, 1), (1, 2), (0, 3)]
        Q = [0.0] * 4
        for i, (f, (a, b)) in enumerate(zip(_equilibrium(s, rho, u, T), s.velocities())):
            cx, cy = s.xi[a] - u[0], s.xi[b] - u[1]
            Q = [q + (F[:, i] - f) * (cx ** m * cy ** n) for q, (m, n) in zip(Q, powers)]
        he = [[1.0, x, (x * x - 1) / 2, (x ** 3 - 3 * x) / 6] for x in s.xi]
        coef = 1.0 / s.tau - 1.0 / ((s.tau - 0.5) / s.pr + 0.5)
        extra = [coef * s.w[a] * s.w[b] * sum(q * (he[a][m] * he[b][n]) for q, (m, n) in zip(Q, powers))
                 for a, b in s.velocities()]
    for i, f in enumerate(_equilibrium(s, rho, u, T)):
        out = F[:, i] - omega * (F[:, i] - f)
        planes.append(out if extra is None else out + extra[i])
    return planes


def _step(s, dep, F):
    S = torch.empty_like(F)
    for i, at in enumerate(dep):
        S[:, i] = at(F[:, i])
    for i, plane in enumerate(_collide(s, S)):
        F[:, i] = plane
    return F


def _gradient(s, case, seed, dep):
    rho, (u, v), T = _flow(case, seed)
    F = torch.stack(list(_equilibrium(s, rho, [u, v], T)), dim=1)
    kept = []
    for _ in range(case["steps"]):
        kept.append(F.cpu())
        F = _step(s, dep, F)
    final = sum(F[0, i] for i in range(s.q))
    lam = torch.zeros_like(F)
    lam[0] = _objective(case, seed)
    for F in reversed(kept):
        F = F.to(lam.device)
        S = torch.stack([at(F[:, i]) for i, at in enumerate(dep)], dim=1).requires_grad_()
        with torch.enable_grad():
            mu, = torch.autograd.grad(torch.stack(_collide(s, S), dim=1), S, lam)
        del S
        for i, at in enumerate(dep):     # the transposed interpolation of one plane
            z = torch.zeros_like(F[:, i]).requires_grad_()
            with torch.enable_grad():
                lam[:, i], = torch.autograd.grad(at(z), z, mu[:, i])
    u, v = u.requires_grad_(), v.requires_grad_()
    du = dv = 0.0
    with torch.enable_grad():
        for i, f in enumerate(_equilibrium(s, rho, [u, v], T)):
            a, b = torch.autograd.grad(f, (u, v), lam[:, i], retain_graph=True)
            du, dv = du + a, dv + b
    return {"rho": final, "du": du, "dv": dv}


def exact(case, seed):
    s = _Setup(case)
    with torch.no_grad():
        dep = _departures(s, _device())
        if case.get("grad"):
            return _gradient(s, case, seed, dep)
        F, w = _state(case, seed).double(), _weights(s)
        full = s.prec == "f64" or s.dim == 3
        if not full:
            for k, i in itertools.product(range(s.npop), range(s.q)):
                F[k, i] += w[k][i]
        for _ in range(case["steps"]):
            F = _step(s, dep, F)
        out = {}
        if case.get("fields"):
            rho, (u, v), T = _moments(s, F)
            out = {"rho": rho, "u": u, "v": v, "T": T, "sums": None}
        if not full:
            for k, i in itertools.product(range(s.npop), range(s.q)):
                F[k, i] -= w[k][i]
        return {**out, "state": F}
