"""The workloads whose speed is watched: what a user has the solver do, through
its public entry points (Solver, Pool and serving.serve, autotune.tune).

A solve is init from the initial fields, n time steps, and the fields back.
Small solves hand over numpy arrays, as the validation runs do; large ones
keep their FP64 fields on the GPU and read them back there, as the benchmark
does.  `tune` picks the launch shape with the autotuner once, when the plan
is made, which is what the benchmark does for its boxes; the others run the
default shape, which is what the validation runs and the pool do.
"""
import decimal
import math

import numpy as np
import torch

from paper_1608_06345_gb300 import autotune, lbm, serving

PERIODIC, OPEN = 0, 1
WORD = {"f64": 8, "f32": 4, "f32_s16f": 2, "f32_s16bf": 2}
FLOPS = {2: 868, 3: 2235}  # per cell and step: moments, equilibria, relaxation of g and h
DIRS = {2: 37, 3: 107}

# kind "solve": step = exact streaming, "fd" = the finite-difference scheme of
# Sec. III at lambda 0.03; "watch": fields and totals of a run in progress;
# "serve": a queue of shock tubes through the pool
BASE = dict(kind="solve", D=2, nx=64, ny=64, nz=1, open_x=False, open_y=False, prec="f32", flow="box", gamma=1.4,
            tau_f=0.55, tau_g=0.7, steps=10, fd=False, tune=False, host=False, requests=0)


def _case(**kw):
    c = dict(BASE)
    c.update(kw)
    return c


def listed():
    return [
        # a unit-test-sized box with ragged rows: launch and latency count
        _case(name="tiny_2d_f32", nx=300, ny=7, steps=40, flow="rough", host=True, tau_f=0.6, tau_g=0.6),
        # the classic Sod tube of the benchmark set, FP64, host arrays in and out
        _case(name="sod_2d_f64", nx=1000, ny=4, open_x=True, prec="f64", flow="sod", steps=500, tau_f=0.6, tau_g=0.6,
              host=True, tune=True),
        # the paper's own 3D validation tube (Sec. V), FP64, the first third of its 180 steps
        _case(name="paper_tube_3d_f64", D=3, nx=1000, ny=16, nz=16, open_x=True, prec="f64", flow="paper", steps=60,
              tau_f=2 / 3, tau_g=2 / 3, host=True),
        # a reference-precision box of the periodic recipe
        _case(name="box_2d_f64", nx=1024, ny=1024, prec="f64", steps=20),
        # the benchmark's headline box
        _case(name="box_2d_f32", nx=4096, ny=4096, steps=128, tune=True),
        # 16-bit storage on a ragged channel (open ends in x)
        _case(name="channel_2d_f16", nx=2999, ny=1777, open_x=True, prec="f32_s16f", steps=40),
        # the benchmark's 3D box
        _case(name="box_3d_f32", D=3, nx=256, ny=256, nz=256, steps=10, tau_f=0.6, tau_g=0.6, tune=True),
        # 3D, 16-bit storage, ragged rows, open ends in y
        _case(name="box_3d_bf16", D=3, nx=193, ny=130, nz=97, open_y=True, prec="f32_s16bf", steps=20, tau_f=0.6,
              tau_g=0.6),
        # the finite-difference scheme on the benchmark's box, and in 3D
        _case(name="fd_2d_f32", nx=4096, ny=4096, steps=20, fd=True),
        _case(name="fd_3d_f32", D=3, nx=112, ny=96, nz=80, steps=10, fd=True, tau_f=0.8, tau_g=0.8),
        # watching a run: the fields and the conserved totals of its present state
        _case(name="watch_2d_f32", kind="watch", nx=2048, ny=2048),
        # serving: a queue of shock tubes of uneven length and step count
        _case(name="serve_2d_f32", kind="serve", nx=12000, ny=4, open_x=True, flow="sod", steps=700, requests=20),
    ]


def draw(rng):
    """One more case of the same ranges, no dearer than the largest listed one."""
    kind = rng.choice(["solve", "solve", "solve", "fd", "watch", "serve"])
    D = 3 if rng.random() < 0.4 and kind != "serve" else 2
    prec = rng.choice(["f64", "f32", "f32", "f32_s16f", "f32_s16bf"])
    tau_f, tau_g = rng.uniform(0.55, 1.0), rng.uniform(0.55, 1.0)
    gamma = rng.uniform(1.1, 1.6)
    if kind == "serve":
        return _case(kind="serve", nx=int(math.exp(rng.uniform(math.log(400), math.log(12000)))), ny=4, open_x=True,
                     prec="f32", flow="sod", steps=rng.randint(150, 700), requests=rng.randint(4, 20), gamma=gamma)
    cells = math.exp(rng.uniform(math.log(1000), math.log(6e6 if D == 2 else 2e6)))
    if prec == "f64":
        cells = min(cells, 1e6)
    ratio = math.exp(rng.uniform(-1.2, 1.2))
    if D == 2:
        nx = max(5, round(math.sqrt(cells) * ratio))
        ny, nz = max(3, round(cells / nx)), 1
    else:
        nx = max(5, round(cells ** (1 / 3) * ratio))
        ny = max(3, round(math.sqrt(cells / nx) * math.exp(rng.uniform(-0.5, 0.5))))
        nz = max(3, round(cells / nx / ny))
    steps = max(1, min(160, int(rng.uniform(0.3, 1.0) * 3e7 / (nx * ny * nz))))
    return _case(kind="watch" if kind == "watch" else "solve", D=D, nx=nx, ny=ny, nz=nz, open_x=rng.random() < 0.4,
                 open_y=rng.random() < 0.3, prec=prec, flow=rng.choice(["box", "box", "rough"]), gamma=gamma,
                 tau_f=max(tau_f, 0.7) if kind == "fd" else tau_f, tau_g=max(tau_g, 0.7) if kind == "fd" else tau_g,
                 steps=min(steps, 40) if kind == "fd" else steps, fd=kind == "fd",
                 tune=D == 2 and kind == "solve" and rng.random() < 0.5, host=nx * ny * nz < 30000)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _shape(case):
    return (case["nx"], case["ny"], case["nz"])[: case["D"]]


def _cells(case):
    return case["nx"] * case["ny"] * case["nz"]


def _bc(case):
    return (OPEN if case["open_x"] else PERIODIC, OPEN if case["open_y"] else PERIODIC, PERIODIC)[: case["D"]]


def _tube(nx, rows, D, left, right):
    """(rho, u, T) of a diaphragm at nx / 2, the same in every row."""
    rho = np.tile(np.where(np.arange(nx) < nx // 2, left[0], right[0]), rows)
    T = np.tile(np.where(np.arange(nx) < nx // 2, left[1], right[1]), rows)
    return rho, np.zeros((D, nx * rows)), T


def _fields(case, seed):
    """(rho, u, T) as float64 CUDA tensors: 8 random Fourier modes of 2 percent
    velocity and 1 percent density and temperature, cell-wise noise of the
    same size, or a shock tube whose states vary a little with the seed."""
    D, N, shape = case["D"], _cells(case), _shape(case)
    rng = np.random.default_rng(seed)
    if case["flow"] in ("sod", "paper"):
        a, b = rng.uniform(0.98, 1.02, 2)
        left, right = ((a, 1.0), (0.125 * b, 0.8)) if case["flow"] == "sod" else ((4 * a, 1.0), (b, 1.0))
        return tuple(torch.from_numpy(f).cuda() for f in _tube(case["nx"], N // case["nx"], D, left, right))
    if case["flow"] == "rough":
        g = torch.Generator(device="cuda").manual_seed(int(seed))
        noise = 0.04 * torch.rand((2 + D, N), generator=g, device="cuda", dtype=torch.float64) - 0.02
        return 1 + noise[0], noise[1:1 + D].contiguous(), 1 + noise[-1]
    axes = [torch.arange(n, device="cuda", dtype=torch.float64) * (2 * math.pi / n) for n in shape]
    rho = torch.ones(N, device="cuda", dtype=torch.float64)
    u = torch.zeros((D, N), device="cuda", dtype=torch.float64)
    T = torch.ones(N, device="cuda", dtype=torch.float64)
    for _ in range(8):
        k = rng.integers(-6, 7, D)
        angle = axes[0] * float(k[0]) + rng.uniform(0, 2 * math.pi)
        for a in range(1, D):
            angle = angle + (axes[a] * float(k[a])).reshape((-1,) + (1,) * a)
        e = rng.normal(size=D)
        wave = torch.cos(angle).reshape(-1)
        for a in range(D):
            u[a] += (0.02 * e[a] / math.sqrt(float(e @ e))) * wave
        rho += (0.01 / 8 * rng.uniform(-1, 1)) * wave
        T += (0.01 / 8 * rng.uniform(-1, 1)) * wave
    return rho, u, T


def _requests(case, seed):
    """Shock tubes of up to case["nx"] cells and case["steps"] steps, each with
    its own gas, relaxation time and reference state."""
    shape_rng, rng = np.random.default_rng(case["requests"]), np.random.default_rng(seed)
    out = []
    for rid in range(case["requests"]):
        nx = int(math.exp(shape_rng.uniform(math.log(256), math.log(case["nx"] + 1))))
        steps = int(shape_rng.integers(case["steps"] // 4, case["steps"] + 1))
        rr, rp = rng.uniform(1.2, 2.5, 2)
        left, right = (math.sqrt(rr), math.sqrt(rp / rr)), (1 / math.sqrt(rr), math.sqrt(rr / rp))
        rho0 = 0.5 * (left[0] + right[0])
        T0 = 0.5 * (left[0] * left[1] + right[0] * right[1]) / rho0
        tau = float(rng.uniform(0.7, 1.0))
        fields = _tube(nx, case["ny"], 2, left, right)
        out.append(serving.Request(rid, (nx, case["ny"]), (OPEN, PERIODIC), float(rng.uniform(1.2, case["gamma"] + 0.2)),
                                   tau, tau, steps, fields, rho0=rho0, T0=T0))
    return out


# ---------------------------------------------------------------------------
# what a program keeps, and one pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    lbm.load()
    if case["kind"] == "serve":
        reqs = _requests(case, seed)
        return dict(case=case, requests=reqs, arrivals=np.zeros(len(reqs)),
                    backend=serving.PoolBackend(lbm.Pool(lbm.LBM_D2Q37, lbm.LBM_F32, budget_bytes=256 << 20)))
    N, D = _cells(case), case["D"]
    fields = _fields(case, seed)
    # the classic tube spans a factor 8 in density: its populations are stored whole
    rho0 = -1.0 if case["flow"] in ("sod", "paper") and case["prec"] in ("f64", "f32") else 0.0
    s = lbm.Solver(lbm.LBM_D2Q37 if D == 2 else lbm.LBM_D3Q107, case["gamma"], case["tau_f"], case["tau_g"],
                   _shape(case), bc=_bc(case), prec=lbm.PREC_NAMES[case["prec"]], rho0=rho0)
    s.init(*fields)
    if case["tune"]:
        autotune.tune(s, reps=5, cache_path=None)
    state = dict(case=case, solver=s)
    if case["kind"] == "watch":
        s.step(3)
    if case["host"]:
        state["fields"] = tuple(f.cpu().numpy() for f in fields)
    else:
        state["fields"] = fields
        state["out"] = tuple(torch.empty((n, N) if n > 1 else N, device="cuda", dtype=torch.float64) for n in (1, D, 1))
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "serve":
        records = serving.serve(state["requests"], state["arrivals"], state["backend"], keep_results=True)
        return [r.result for r in records]
    s = state["solver"]
    if case["kind"] != "watch":
        s.init(*state["fields"])
        if case["fd"]:
            s.step_fd(case["steps"], 0.03)
        else:
            s.step(case["steps"])
    if case["host"]:
        out = s.moments()
    else:
        out = state["out"]
        s.moments_device(*out)
    if case["kind"] == "watch":
        return {"fields": out, "totals": s.conserved()}
    return out


def work(case):
    """A step reads and writes each of the 2Q populations of a cell once; a
    solve also reads the initial fields and writes the final ones."""
    D, word = case["D"], WORD[case["prec"]]
    if case["kind"] == "serve":
        reqs = _requests(case, 0)
        updates, cells = sum(r.cells * r.steps for r in reqs), sum(r.cells for r in reqs)
    else:
        cells = _cells(case)
        updates = cells * case["steps"]
    pops, fields = 2 * DIRS[D] * word, 8 * (D + 2)
    if case["kind"] == "watch":
        return {"bytes": cells * (pops + fields), "flops": cells * 12 * DIRS[D]}
    return {"bytes": updates * 2 * pops + cells * 2 * fields, "flops": updates * FLOPS[D]}


# ---------------------------------------------------------------------------
# the same in 64 bits: Eq. (14)-(18) in plain torch
# ---------------------------------------------------------------------------
_GROUPS = {2: [(0, 0), (1, 0), (1, 1), (2, 0), (2, 1), (3, 0), (3, 1), (3, 3)],
           3: [(0, 0, 0), (1, 0, 0), (1, 1, 0), (1, 1, 1), (2, 0, 0), (2, 1, 1), (2, 2, 0), (2, 2, 2), (3, 0, 0),
               (3, 1, 1)]}
_MOMENTS = {2: [(0, 0), (2, 0), (4, 0), (2, 2), (6, 0), (4, 2), (6, 2), (4, 4), (8, 0)],
            3: [(0, 0, 0), (2, 0, 0), (4, 0, 0), (2, 2, 0), (6, 0, 0), (4, 2, 0), (2, 2, 2), (6, 2, 0), (4, 4, 0),
                (4, 2, 2), (8, 0, 0)]}
_tables = {}


def _table(D):
    """Velocities c[Q, D], weights w[Q] and scale r (xi = r c) of Tables I and
    II: the moments of the unit Gaussian up to degree 8, solved for the group
    weights at a given r, with r where the last moment holds too."""
    if D in _tables:
        return _tables[D]
    span = range(-3, 4)
    every = [(x, y) for x in span for y in span] if D == 2 else [(x, y, z) for x in span for y in span for z in span]
    groups = [[c for c in every if tuple(sorted(map(abs, c), reverse=True)) == g] for g in _GROUPS[D]]
    with decimal.localcontext() as ctx:
        ctx.prec = 60
        dec = decimal.Decimal

        def row(e):
            return [dec(sum(math.prod(v ** p for v, p in zip(c, e)) for c in g)) for g in groups]

        def moment(e, r2):
            return dec(math.prod(math.prod(range(p - 1, 0, -2)) for p in e)) / r2 ** (sum(e) // 2)

        def weights(r2):
            a = [row(e) + [moment(e, r2)] for e in _MOMENTS[D][:-1]]
            n = len(a)
            for k in range(n):
                p = max(range(k, n), key=lambda i: abs(a[i][k]))
                a[k], a[p] = a[p], a[k]
                a[k] = [v / a[k][k] for v in a[k]]
                for i in range(n):
                    if i != k and a[i][k]:
                        a[i] = [x - a[i][k] * y for x, y in zip(a[i], a[k])]
            w = [r[-1] for r in a]
            last = _MOMENTS[D][-1]
            return w, sum(x * y for x, y in zip(w, row(last))) - moment(last, r2)

        lo, hi = dec("1.4327"), dec("1.4328")  # r^2 near 1.19698^2
        flo, fhi = weights(lo)[1], weights(hi)[1]
        for _ in range(12):
            if fhi == flo:
                break
            lo, hi, flo = hi, hi - fhi * (hi - lo) / (fhi - flo), fhi
            fhi = weights(hi)[1]
        w, r = weights(hi)[0], float(hi.sqrt())
    c = np.array([v for g in groups for v in g])
    _tables[D] = c, np.array([float(x) for x, g in zip(w, groups) for _ in g]), r
    return _tables[D]


class _Exact:
    def __init__(self, D, shape, bc, gamma, tau_f, tau_g):
        c, w, r = _table(D)
        self.D, self.shape, self.bc, self.c, self.r = D, tuple(shape), bc, c, r
        self.delta, self.tau_f, self.tau_g = 2 / (gamma - 1) - D, tau_f, tau_g
        self.N = math.prod(shape)
        self.xi = torch.from_numpy(r * c.astype(float)).cuda()
        self.w = torch.from_numpy(w).cuda()[:, None]
        self.x2 = (self.xi ** 2).sum(1)[:, None]
        self.whole, self.pull = {}, torch.empty(0)

    def equilibrium(self, rho, u, T):
        D, x2 = self.D, self.x2
        s, u2, t = self.xi @ u, (u ** 2).sum(0), T - 1
        F = 1 + s + (s * s - u2 + t * (x2 - D)) / 2
        F += s * (s * s - 3 * u2 + 3 * t * (x2 - D - 2)) / 6
        F += (s ** 4 - 6 * s * s * u2 + 3 * u2 * u2 + 6 * t * (s * s * (x2 - D - 4) + (D + 2 - x2) * u2)
              + 3 * t * t * (x2 * x2 - 2 * (D + 2) * x2 + D * (D + 2))) / 24
        return F.mul_(self.w * rho)

    def chunks(self):
        n = 1 << 21 if self.D == 2 else 1 << 20
        return [slice(k, min(k + n, self.N)) for k in range(0, self.N, n)]

    def init(self, rho, u, T):
        self.g = torch.empty((len(self.c), self.N), device="cuda", dtype=torch.float64)
        self.h = torch.empty_like(self.g)
        for k in self.chunks():
            self.g[:, k] = self.equilibrium(rho[k], u[:, k], T[k])
            self.h[:, k] = self.delta / 2 * T[k] * self.g[:, k]

    def moments(self, g, h):
        rho = g.sum(0)
        u = (self.xi.T @ g) / rho
        E = ((self.x2 / 2 * g).sum(0) + h.sum(0)) / rho
        return rho, u, 2 * (E - (u ** 2).sum(0) / 2) / (self.D + self.delta)

    def shifted(self, q, by):
        """Every cell's value at its place minus `by`, wrapped or the edge cell's."""
        if by not in self.whole:
            at = torch.zeros(1, device="cuda", dtype=torch.int64)
            for a in reversed(range(self.D)):
                n = self.shape[a]
                p = torch.arange(n, device="cuda") - by[a]
                p = p % n if self.bc[a] == PERIODIC else p.clamp(0, n - 1)
                at = at[..., None] * n + p
            self.whole = {} if self.N > 1 << 20 else self.whole
            self.whole[by] = at.reshape(-1)
        return q[self.whole[by]]

    def step(self, fd):
        if not fd and self.N <= 1 << 16:  # a small grid: all directions at once
            if not self.pull.numel():
                here = torch.arange(self.N, device="cuda")
                self.pull = torch.stack([self.shifted(here, tuple(c)) for c in self.c.tolist()])
            g, h = self.g.gather(1, self.pull), self.h.gather(1, self.pull)
        else:
            g, h = torch.empty_like(self.g), torch.empty_like(self.h)
        for i, c in enumerate(self.c.tolist() if fd or self.N > 1 << 16 else []):
            for q, new in ((self.g, g), (self.h, h)):
                if not fd:
                    new[i] = self.shifted(q[i], tuple(c))
                    continue
                new[i] = q[i]
                for a in range(self.D):
                    if c[a]:
                        s = 1 if c[a] > 0 else -1
                        m2, m1, p1 = (self.shifted(q[i], tuple(s * k if b == a else 0 for b in range(self.D)))
                                      for k in (2, 1, -1))
                        new[i] -= 0.03 * self.r * c[a] * s / 6 * (m2 - 6 * m1 + 3 * q[i] + 2 * p1)
        for k in self.chunks():
            gk, hk = (self.g[:, k], self.h[:, k]) if fd else (g[:, k], h[:, k])
            rho, u, T = self.moments(gk, hk)
            F = self.equilibrium(rho, u, T)
            g[:, k] += (F - gk) / self.tau_f
            h[:, k] += (self.delta / 2 * T * F - hk) / self.tau_g
        self.g, self.h = g, h

    def fields(self):
        parts = [self.moments(self.g[:, k], self.h[:, k]) for k in self.chunks()]
        return tuple(torch.cat([p[j] for p in parts], dim=-1) for j in range(3))


def exact(case, seed):
    if case["kind"] == "serve":
        out = []
        for r in _requests(case, seed):
            # a tube is the same in each of its rows
            e = _Exact(2, (r.shape[0], 1), r.bc, r.gamma, r.tau_f, r.tau_g)
            e.init(*(torch.from_numpy(np.ascontiguousarray(f[..., : r.shape[0]])).cuda() for f in r.fields))
            for _ in range(r.steps):
                e.step(False)
            out.append(tuple(f.repeat((1,) * (f.dim() - 1) + (r.shape[1],)) for f in e.fields()))
        return out
    rows = _cells(case) // case["nx"]
    tube = case["flow"] in ("sod", "paper")
    shape = (case["nx"],) + (1,) * (case["D"] - 1) if tube else _shape(case)
    e = _Exact(case["D"], shape, _bc(case), case["gamma"], case["tau_f"], case["tau_g"])
    e.init(*(f[..., : e.N].contiguous() for f in _fields(case, seed)))
    for _ in range(3 if case["kind"] == "watch" else case["steps"]):
        e.step(case["fd"])
    rho, u, T = (f.repeat((1,) * (f.dim() - 1) + (rows,)) if tube else f for f in e.fields())
    if case["kind"] != "watch":
        return rho, u, T
    mass, energy = e.g.sum(), (e.x2 / 2 * e.g).sum() + e.h.sum()
    return {"fields": (rho, u, T), "totals": torch.stack([mass, *(e.xi.T @ e.g.sum(1)), energy])}
