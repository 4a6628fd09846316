"""The work that users of this library have it do, as timed cases.

One layer: w_t = -J(psi, w) - J(psi, y)/Ro + lap(w)/Re + F on [0, 1] x [-1, 1],
psi the prolonged solution of lap(psibar) = R w on the elliptic grid; two
layers: the coupled equations of the stratified basin.  A pass goes through
the public calls of paper_1308_3290_gb300.qg and .adjoint, from the state a
program has on the GPU to the fields it reads back.

Grids are powers of two, as the library requires; the "odd" sizes of the range
are its other aspect ratios (square, wide and very tall basins, whose spacings
differ in x and y).
"""
import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_1308_3290_gb300 import adjoint, qg

DTYPES = {"f32": torch.float32, "f64": torch.float64}
ESZ = {"f32": 4, "f64": 8}
RO = 0.0016                    # Experiment I; Re = 200
TWO = dict(Ro=2.49e-4, Fr=0.087, delta=0.2, sigma=1.43e-3)   # the two-layer experiment, Re = 697.16


def listed():
    def basin(name, nx, ny, levels, dtype, steps, **kw):
        return dict(name=name, kind="basin", nx=nx, ny=ny, levels=levels, dtype=dtype, steps=steps,
                    Re=200.0, layers=1, **kw)

    return [
        # one handle-free solve of a small grid: the shortest call, all latency
        dict(name="poisson_noalloc_64x128_f32", kind="noalloc", nx=64, ny=128, dtype="f32"),
        # the paper's own basin in double precision: a long run of launch-bound steps
        basin("basin_64x128_l1_f64", 64, 128, 1, "f64", 50),
        # the size of the time-mean study and of the adjoint, in single precision
        basin("basin_256x512_l1_f32", 256, 512, 1, "f32", 50),
        # a wide basin run as a production segment: adaptive step, time means, diagnostics
        dict(name="segment_1024x512_l1_f32", kind="segment", nx=1024, ny=512, levels=1, dtype="f32",
             steps=20, Re=312.5),
        # the headline basin: two levels of coarsening
        basin("basin_2048x4096_l2_f32", 2048, 4096, 2, "f32", 20),
        # the standard full-grid solver the paper compares with
        basin("basin_2048x4096_l0_f32", 2048, 4096, 0, "f32", 8),
        # a double-precision control run without coarsening
        basin("basin_1024x2048_l0_f64", 1024, 2048, 0, "f64", 3),
        # the stratified basin, both layers coupled in the elliptic solve
        dict(name="two_layer_1024x2048_l1_f32", kind="basin", nx=1024, ny=2048, levels=1, dtype="f32",
             steps=20, Re=697.16, layers=2),
        # an ensemble of uneven basins (128 x 256 to 1024 x 2048), one launch per step
        dict(name="ensemble_48_f32", kind="ensemble", members=48, big=4, dtype="f32", steps=6),
        # gradient of the mean kinetic energy with respect to the wind field, checkpointed
        dict(name="adjoint_256x512_l1_f32", kind="adjoint", nx=256, ny=512, levels=1, dtype="f32",
             steps=40, first=20, every=10),
        # the operators called one by one: restriction, elliptic solve, prolongation
        dict(name="operators_2048x1024_l1_f32", kind="operators", nx=2048, ny=1024, levels=1, dtype="f32"),
        # the paper's other elliptic solver, V-cycles on the coarse grid
        dict(name="multigrid_1024x2048_l1_f32", kind="multigrid", nx=1024, ny=2048, levels=1, dtype="f32",
             steps=3, cycles=3, Re=200.0),
    ]


def draw(rng):
    kind = rng.choice(["basin"] * 6 + ["segment", "ensemble", "adjoint", "operators", "multigrid", "noalloc"])
    dtype = rng.choice(["f32", "f32", "f32", "f64"])
    if kind == "ensemble":
        return dict(kind=kind, members=rng.randint(5, 40), big=rng.randint(2, 4), dtype="f32", steps=rng.randint(1, 6))
    while True:
        nx = 2 ** rng.randint(6, 11)
        ny = int(nx * rng.choice([0.5, 1, 2, 2, 2, 4]))
        levels = rng.choice([0, 1, 1, 2, 2, 3])
        layers = 2 if kind == "basin" and rng.random() < 0.25 else 1
        if kind == "noalloc":
            return dict(kind=kind, nx=2 ** rng.randint(4, 8), ny=2 ** rng.randint(4, 9), dtype=dtype)
        if kind == "adjoint":
            nx = 2 ** rng.randint(6, 9)
            steps = rng.randint(8, 40)
            return dict(kind=kind, nx=nx, ny=nx * 2, levels=rng.randint(0, 2), dtype=dtype, steps=steps,
                        first=rng.randint(0, steps - 1), every=rng.choice([1, 4, 10]))
        if kind == "operators":
            return dict(kind=kind, nx=nx, ny=min(ny, 4096), levels=max(1, levels), dtype=dtype)
        Re = round(rng.uniform(200.0, 1000.0), 1)
        if kind == "multigrid":
            return dict(kind=kind, nx=min(nx, 1024), ny=2 * min(nx, 1024), levels=min(levels, 2), dtype=dtype,
                        steps=rng.randint(1, 3), cycles=rng.randint(2, 4), Re=Re)
        steps = rng.randint(2, 40)
        c = dict(kind=kind, nx=nx, ny=ny, levels=levels, dtype=dtype, steps=steps, Re=Re)
        if kind == "basin":
            c["layers"] = layers
        # no more work than the largest listed case: 8 full-grid FP32 steps of
        # 2048 x 4096 (double precision counted 16 times: its units are that few)
        cost = nx * ny * layers * steps * (16 if dtype == "f64" else 1)
        if ny <= 4096 and nx >= 64 and min(nx, ny) >> levels >= 8 and cost <= 8 * 2048 * 4096:
            return c


# ---- what a program has in hand before the call ------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _gyre(nx, ny, seed, dtype, amp=200.0):
    """A spun-up looking vorticity field: four cells with a western boundary
    concentration, mesoscale modes and grid-scale noise."""
    g = _gen(seed)
    d = dict(dtype=torch.float64, device="cuda")
    x = (torch.arange(1, nx, **d) / nx)[None, :]
    y = (torch.arange(1, ny, **d) / ny)[:, None]
    f = amp * torch.exp(-x / 0.05) * torch.sin(2 * math.pi * y)
    f = f + 0.2 * amp * torch.sin(math.pi * x) * torch.sin(4 * math.pi * y)
    k = torch.randint(2, 24, (12, 2), generator=g, device="cuda").double()
    a = torch.randn(12, generator=g, **d) * 0.05 * amp
    for i in range(12):
        f = f + a[i] * torch.sin(math.pi * k[i, 0] * x) * torch.sin(math.pi * k[i, 1] * y)
    f = f + 0.1 * torch.randn(ny - 1, nx - 1, generator=g, **d)
    return f.to(DTYPES[dtype]).contiguous()


def _wind(nx, ny, seed, dtype):
    """sin(pi y)/Ro with a smooth perturbation: the control of the adjoint."""
    g = _gen(seed)
    d = dict(dtype=torch.float64, device="cuda")
    x = (torch.arange(1, nx, **d) / nx)[None, :]
    y = (torch.arange(1, ny, **d) / ny)[:, None]
    f = torch.sin(math.pi * (2 * y - 1)).expand(ny - 1, nx - 1).clone()
    a = torch.randn(4, 4, generator=g, **d) * 0.05
    for k in range(4):
        for l in range(4):
            f += a[k, l] * torch.sin((k + 1) * math.pi * x) * torch.sin((l + 1) * math.pi * y)
    return (f / RO).to(DTYPES[dtype]).contiguous()


def _dt(c):
    """A step within the advective and viscous limits of the finer spacing;
    the cap of the adaptive step lies above what the flow then allows."""
    return (2e-2 if c["kind"] == "segment" else 4e-3) / max(c["nx"], c["ny"] / 2)


def _members(c, seed):
    """Sizes, levels and parameters of the ensemble: a fixed mix of sizes
    (the seed moves only the flow parameters and the states)."""
    sizes = [(128 << k, 256 << k) for k in range(c["big"])]
    g = np.random.default_rng(seed)
    out = []
    for i in range(c["members"]):
        nx, ny = sizes[(i * 5 + i // 3) % len(sizes)]
        out.append(dict(nx=nx, ny=ny, Re=float(g.uniform(200, 1000)), Ro=RO, levels=1 + (i // 2) % 2,
                        dt=4e-3 / 1024, amp=float(g.uniform(0.5, 1.5))))
    return out


def prepare(c, seed):
    s = {"c": c, "kind": c["kind"]}
    if c["kind"] == "noalloc":
        s["rhs"] = _gyre(c["nx"], c["ny"], seed, c["dtype"])
        s["out"] = torch.empty_like(s["rhs"])
        return s
    if c["kind"] == "ensemble":
        m = _members(c, seed)
        s["e"] = qg.Ensemble(m, dtype=c["dtype"])
        s["w"] = [_gyre(x["nx"], x["ny"], seed * 1000 + i, c["dtype"]) for i, x in enumerate(m)]
        return s
    nx, ny = c["nx"], c["ny"]
    if c.get("layers") == 2:
        s["b"] = qg.Basin(nx, ny, Re=c["Re"], levels=c["levels"], dt=_dt(c), dtype=c["dtype"], layers=2,
                          y0=-0.5, y1=0.5, **TWO)
        s["w"] = [_gyre(nx, ny, 2 * seed + k, c["dtype"], amp=(0.5, 0.1)[k]) for k in (0, 1)]
        return s
    s["b"] = qg.Basin(nx, ny, Re=c.get("Re", 200.0), Ro=RO, levels=c["levels"], dt=_dt(c), dtype=c["dtype"])
    s["w"] = _gyre(nx, ny, seed, c["dtype"])
    if c["kind"] == "segment":
        qg.qg_set_cfl(s["b"].h, 0.5)
    if c["kind"] == "multigrid":
        qg.qg_set_solver(s["b"].h, qg.QG_SOLVER_MULTIGRID, c["cycles"])
    if c["kind"] == "adjoint":
        s["F"] = _wind(nx, ny, seed, c["dtype"])
    if c["kind"] == "operators":
        l = c["levels"]
        s["coarse"] = _gyre(nx >> l, ny >> l, seed + 1, c["dtype"], amp=1.0)
    return s


# ---- one pass ----------------------------------------------------------------

def run(s):
    c, kind = s["c"], s["kind"]
    if kind == "noalloc":
        nx, ny = c["nx"], c["ny"]
        qg.qg_poisson_solve_noalloc(nx, ny, 1.0 / nx, 2.0 / ny, qg.QG_F32 if c["dtype"] == "f32" else qg.QG_F64,
                                    s["rhs"], s["out"], torch.cuda.current_stream().cuda_stream)
        return s["out"]
    if kind == "ensemble":
        e = s["e"]
        for i, w in enumerate(s["w"]):
            e.member(i).set_state(w)
        e.step(c["steps"])
        return [e.member(i).state() for i in range(len(e))]
    b = s["b"]
    if kind == "operators":
        wc = b.restrict(s["w"], c["levels"])
        return [wc, b.poisson_solve(wc, c["levels"]), b.prolong(s["coarse"], c["levels"])]
    if kind == "adjoint":
        F = s["F"].detach().requires_grad_(True)
        J = adjoint.mean_kinetic_energy(F, b, s["w"], c["steps"], c["first"], c["every"])
        J.backward()
        return [J.detach().to(F.dtype), F.grad]
    if kind == "segment":
        b.set_state(s["w"])
        qg.qg_stats_begin(b.h)
        b.step(c["steps"])
        mp, mq = torch.empty_like(s["w"]), torch.empty_like(s["w"])
        qg.qg_stats_mean_psi(b.h, mp)
        qg.qg_stats_mean_q(b.h, mq)
        qg.qg_stats_end(b.h)
        # a basin's energy, enstrophy and largest velocity are as good as its fields
        num = [s["w"].new_tensor(v, device="cpu") for v in b.diagnostics()]
        return [b.state(), mp, mq, num]
    if c.get("layers") == 2:
        for k in (0, 1):
            b.set_state(s["w"][k], k)
        b.step(c["steps"])
        return [b.state(0), b.state(1), b.psi(0), b.psi(1)]
    b.set_state(s["w"])
    b.step(c["steps"])
    return [b.state(), b.psi()]


# ---- what a pass cannot do without --------------------------------------------

def _step_work(nx, ny, levels, layers, esz):
    """(bytes, flops) of one step: each stage reads the state, writes it, and
    from the second on reads the step's first state; the elliptic grid's
    right-hand side and solution pass through the three sweeps of the sine
    transforms.  Flops: 45 a fine node and stage; two transforms in each
    direction of 2.5 N log2 N."""
    n, m = nx * ny * layers, (nx >> levels) * (ny >> levels) * layers
    byt = esz * (8 * n + (3 * n if levels == 0 else 6 * m) + 18 * m)
    flops = 3 * (45 * n + m * 5 * (math.log2(nx >> levels) + math.log2(ny >> levels)))
    return byt, flops


def work(c):
    esz = ESZ[c["dtype"]]
    if c["kind"] == "ensemble":
        got = [_step_work(m["nx"], m["ny"], m["levels"], 1, esz) for m in _members(c, 0)]
        return {"bytes": c["steps"] * sum(g[0] for g in got), "flops": c["steps"] * sum(g[1] for g in got)}
    nx, ny = c["nx"], c["ny"]
    n = nx * ny
    lg = 5 * (math.log2(nx) + math.log2(ny))
    if c["kind"] == "noalloc":
        return {"bytes": 2 * esz * n, "flops": n * lg}
    m = n >> 2 * c["levels"]
    if c["kind"] == "operators":
        return {"bytes": esz * (2 * n + 4 * m), "flops": m * lg + 20 * n}
    byt, flops = _step_work(nx, ny, c["levels"], c.get("layers", 1), esz)
    if c["kind"] == "adjoint":
        # forward, the stages once more in reverse, and their transposes
        return {"bytes": 3 * c["steps"] * byt, "flops": 3 * c["steps"] * flops}
    return {"bytes": c["steps"] * byt, "flops": c["steps"] * flops}


# ---- the same in 64 bits, in plain torch ----------------------------------------

def _dst(f, dim):
    """sum_n f_n sin(pi n k / N) along dim (interior nodes)."""
    f = f.movedim(dim, -1)
    z = torch.zeros(f.shape[:-1] + (1,), dtype=f.dtype, device=f.device)
    ext = torch.cat([z, f, z, -f.flip(-1)], -1)
    return (torch.fft.rfft(ext).imag[..., 1:f.shape[-1] + 1] * -0.5).movedim(-1, dim)


def _eig(mx, my, dx, dy):
    d = dict(dtype=torch.float64, device="cuda")
    lx = -4 * torch.sin(math.pi * torch.arange(1, mx, **d) / (2 * mx)) ** 2 / dx ** 2
    ly = -4 * torch.sin(math.pi * torch.arange(1, my, **d) / (2 * my)) ** 2 / dy ** 2
    return ly[:, None] + lx[None, :]


def _solve(f, dx, dy):
    my, mx = f.shape[0] + 1, f.shape[1] + 1
    fh = _dst(_dst(f, 0), 1) / _eig(mx, my, dx, dy) * (4.0 / mx / my)
    return _dst(_dst(fh, 0), 1)


def _pad(f):
    return torch.nn.functional.pad(f, (1, 1, 1, 1))


def _restrict(f, levels):
    for _ in range(levels):
        f = (f[1:-1:2] * 2 + f[:-2:2] + f[2::2]) / 4
        f = (f[:, 1:-1:2] * 2 + f[:, :-2:2] + f[:, 2::2]) / 4
    return f


def _prolong(f, levels):
    for _ in range(levels):
        for dim in (0, 1):
            p = _pad(f).movedim(dim, 0)[:, 1:-1]
            mid = (p[1:] + p[:-1]) / 2
            # mid, node, mid, ..., node, mid
            f = torch.cat([mid[:1], torch.stack([p[1:-1], mid[1:]], 1).flatten(0, 1)], 0).movedim(0, dim)
    return f


class _Model:
    def __init__(self, nx, ny, Re, levels, dt, amp=1.0, layers=1, F=None, cfl=0.0):
        self.nx, self.ny, self.levels, self.dt, self.cfl = nx, ny, levels, dt, cfl
        self.dx, self.dy = 1.0 / nx, (2.0 if layers == 1 else 1.0) / ny
        d = dict(dtype=torch.float64, device="cuda")
        self.layers, self.Ro, self.Re = layers, RO if layers == 1 else TWO["Ro"], Re
        y = (-1.0 if layers == 1 else -0.5) + self.dy * torch.arange(0, ny + 1, **d)
        self.Y = y[:, None].expand(ny + 1, nx + 1)
        wind = amp * (torch.sin(math.pi * y) / RO if layers == 1 else torch.sin(2 * math.pi * y))
        self.F = wind[1:-1, None].expand(ny - 1, nx - 1) if F is None else F

    def psi(self, w):
        f = 2 ** self.levels
        if self.layers == 1:
            return _prolong(_solve(_restrict(w, self.levels), f * self.dx, f * self.dy), self.levels)
        q = [_restrict(x, self.levels) for x in w]
        my, mx = q[0].shape[0] + 1, q[0].shape[1] + 1
        h = [_dst(_dst(x, 0), 1) * (4.0 / mx / my) for x in q]
        a = self.Ro * _eig(mx, my, f * self.dx, f * self.dy)
        f1, f2 = TWO["Fr"] / TWO["delta"], TWO["Fr"] / (1 - TWO["delta"])
        den = a * (a - f1 - f2)
        p = [(a * h[0] - f2 * h[0] - f1 * h[1]) / den, (a * h[1] - f2 * h[0] - f1 * h[1]) / den]
        return [_prolong(_dst(_dst(x, 0), 1), self.levels) for x in p]

    def jac(self, p, q):
        """Arakawa's Jacobian of two node arrays at the interior nodes."""
        def s(a, i, j):
            return a[1 + j:a.shape[0] - 1 + j, 1 + i:a.shape[1] - 1 + i]
        j1 = (s(p, 1, 0) - s(p, -1, 0)) * (s(q, 0, 1) - s(q, 0, -1)) - (s(p, 0, 1) - s(p, 0, -1)) * (s(q, 1, 0) - s(q, -1, 0))
        j2 = (s(q, 0, 1) * (s(p, 1, 1) - s(p, -1, 1)) - s(q, 0, -1) * (s(p, 1, -1) - s(p, -1, -1))
              - s(q, 1, 0) * (s(p, 1, 1) - s(p, 1, -1)) + s(q, -1, 0) * (s(p, -1, 1) - s(p, -1, -1)))
        j3 = (s(p, 1, 0) * (s(q, 1, 1) - s(q, 1, -1)) - s(p, -1, 0) * (s(q, -1, 1) - s(q, -1, -1))
              - s(p, 0, 1) * (s(q, 1, 1) - s(q, -1, 1)) + s(p, 0, -1) * (s(q, 1, -1) - s(q, -1, -1)))
        return (j1 + j2 + j3) / (12 * self.dx * self.dy)

    def lap(self, f):
        c = f[1:-1, 1:-1]
        return (f[1:-1, 2:] - 2 * c + f[1:-1, :-2]) / self.dx ** 2 + (f[2:, 1:-1] - 2 * c + f[:-2, 1:-1]) / self.dy ** 2

    def rhs(self, w, psi):
        if self.layers == 1:
            p, q = _pad(psi), _pad(w)
            return -self.jac(p, q) - self.jac(p, self.Y) / self.Ro + self.lap(q) / self.Re + self.F
        f1, f2 = TWO["Fr"] / TWO["delta"], TWO["Fr"] / (1 - TWO["delta"])
        v = [(w[0] - f1 * (psi[1] - psi[0])) / self.Ro, (w[1] - f2 * (psi[0] - psi[1])) / self.Ro]
        A = self.Ro / self.Re
        g = [-self.jac(_pad(psi[k]), _pad(w[k])) - self.jac(_pad(psi[k]), self.Y) + A * self.lap(_pad(v[k])) for k in (0, 1)]
        return torch.stack([g[0] + self.F, g[1] - TWO["sigma"] * v[1]])

    def umax(self, psi):
        p = _pad(psi)
        return max(float((p[1:-1, 2:] - p[1:-1, :-2]).abs().max()) / (2 * self.dx),
                   float((p[2:, 1:-1] - p[:-2, 1:-1]).abs().max()) / (2 * self.dy))

    def step(self, w, psi=None):
        dt, u = self.dt, w
        for s, (a, b) in enumerate(((0.0, 1.0), (0.75, 0.25), (1 / 3, 2 / 3))):
            p = psi if s == 0 and psi is not None else self.psi(u)
            if s == 0 and self.cfl:
                dt = min(dt, self.cfl * min(self.dx, self.dy) / self.umax(p))
            u = a * w + b * (u + dt * self.rhs(u, torch.stack(p) if isinstance(p, list) else p))
        return u

    def energy(self, psi):
        p = _pad(psi)
        ex, ey = (p[:, 1:] - p[:, :-1]) / self.dx, (p[1:] - p[:-1]) / self.dy
        return 0.5 * self.dx * self.dy * ((ex * ex).sum() + (ey * ey).sum())


def exact(c, seed):
    kind = c["kind"]
    if kind == "noalloc":
        return _solve(_gyre(c["nx"], c["ny"], seed, c["dtype"]).double(), 1.0 / c["nx"], 2.0 / c["ny"])
    if kind == "ensemble":
        out = []
        for i, m in enumerate(_members(c, seed)):
            M = _Model(m["nx"], m["ny"], m["Re"], m["levels"], m["dt"], amp=m["amp"])
            w = _gyre(m["nx"], m["ny"], seed * 1000 + i, c["dtype"]).double()
            for _ in range(c["steps"]):
                w = M.step(w)
            out.append(w)
        return out
    nx, ny, l = c["nx"], c["ny"], c["levels"]
    if kind == "operators":
        wc = _restrict(_gyre(nx, ny, seed, c["dtype"]).double(), l)
        k = _gyre(nx >> l, ny >> l, seed + 1, c["dtype"], amp=1.0).double()
        return [wc, _solve(wc, 2 ** l / nx, 2 ** l * 2 / ny), _prolong(k, l)]
    if c.get("layers") == 2:
        M = _Model(nx, ny, c["Re"], l, _dt(c), layers=2)
        w = torch.stack([_gyre(nx, ny, 2 * seed + k, c["dtype"], amp=(0.5, 0.1)[k]).double() for k in (0, 1)])
        for _ in range(c["steps"]):
            w = M.step(w)
        return [w[0], w[1]] + M.psi(w)
    w = _gyre(nx, ny, seed, c["dtype"]).double()
    if kind == "adjoint":
        F = _wind(nx, ny, seed, c["dtype"]).double().requires_grad_(True)
        M = _Model(nx, ny, 200.0, l, _dt(c), F=F)
        # torch differentiates the 64-bit steps; each step is recomputed in
        # the reverse sweep, so that only its state is kept
        ckpt = torch.utils.checkpoint.checkpoint
        J = 0.0
        for n in range(c["steps"] + 1):
            if n >= c["first"]:
                J = J + ckpt(lambda u: M.energy(M.psi(u)), w, use_reentrant=False)
            if n < c["steps"]:
                w = ckpt(M.step, w, use_reentrant=False)
        J = J / (c["steps"] - c["first"] + 1)
        J.backward()
        return [J.detach(), F.grad]
    M = _Model(nx, ny, c["Re"], l, _dt(c), cfl=0.5 if kind == "segment" else 0.0)
    if kind == "segment":
        mp, mq = torch.zeros_like(w), torch.zeros_like(w)
        y = M.Y[1:-1, :1]
        for _ in range(c["steps"]):
            p = M.psi(w)
            mp += p / c["steps"]
            mq += (RO * w + y) / c["steps"]
            w = M.step(w, p)
        p = M.psi(w)
        num = [M.energy(p), 0.5 * M.dx * M.dy * (w * w).sum(), torch.tensor(M.umax(p), dtype=torch.float64)]
        return [w, mp, mq, num]
    # (the V-cycles approach the discrete solution, which is what is given here)
    for _ in range(c["steps"]):
        w = M.step(w)
    return [w, M.psi(w)]
