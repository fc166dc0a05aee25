"""Measured cases of the coupled pressure-temperature framework.

A case is one call sequence a program makes every time step (or once per
request): set-up and solve of the coupled system on uniform 2D, axisymmetric
and 3D grids, many problems in one batch, a refined-patch solve, the momentum
predictor and the steps around the solve.  Fields are the repository's
synthetic bubbles (a tanh volume fraction, water and air, dt = 1e-7 over a unit
domain; the stiff regime is the 6.4 mm domain with dt = 1e-5), made on the GPU
from a seed.

    listed()             the cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  inputs, handle and kernel choices on the GPU
    run(state)           one pass through the public entry points
    work(case)           bytes and flops one pass cannot do without
    exact(case, seed)    run's outputs from plain torch in 64 bits
"""
import math

import numpy as np
import torch

from paper_2206_11294_gb300 import autotune, binding, inputs

# Kernel choices are measured once per hierarchy shape and kept, as a program
# that solves many steps or requests of a shape does (autotune.TuningTable).
TABLE = autotune.TuningTable()

WALL, DIRICHLET, AXIS = inputs.BC_WALL, inputs.BC_DIRICHLET, inputs.BC_AXIS


def listed():
    return [
        # the smallest call: one bubble on 64^2, where launches and host waits are the cost
        dict(name="solve_64_fp64", kind="solve", geom="plane", n0=64, n1=64, n2=1, bubbles=1, precision="fp64",
             stiff=False, tuned=False),
        # the benchmark's plane problem in both precisions, kernel choices measured as its time loop does
        dict(name="solve_1024_fp64", kind="solve", geom="plane", n0=1024, n1=1024, n2=1, bubbles=16, precision="fp64",
             stiff=False, tuned=True),
        dict(name="solve_1024_mixed", kind="solve", geom="plane", n0=1024, n1=1024, n2=1, bubbles=16,
             precision="mixed", stiff=False, tuned=True),
        # the benchmark's axisymmetric problem with the library's default kernel choices
        dict(name="solve_axi_512x1024_fp64", kind="solve", geom="axi", n0=512, n1=1024, n2=1, bubbles=1,
             precision="fp64", stiff=False, tuned=False),
        # the largest: a bubble near a rigid wall in 3D, five pressure boundaries
        dict(name="solve_wall3d_256_fp64", kind="solve", geom="wall3d", n0=256, n1=256, n2=256, bubbles=1,
             precision="fp64", stiff=False, tuned=False),
        # a 3D serving request: mixed precision, an odd coarsest grid (5 x 5 x 5)
        dict(name="solve_wall3d_160_mixed", kind="solve", geom="wall3d", n0=160, n1=160, n2=160, bubbles=1,
             precision="mixed", stiff=False, tuned=False),
        # a ragged size with a large coarsest grid (31 x 23 cells, solved from its factors)
        dict(name="solve_992x736_fp64", kind="solve", geom="plane", n0=992, n1=736, n2=1, bubbles=8,
             precision="fp64", stiff=False, tuned=False),
        # many cycles per set-up: the collapse scale, where the coarse levels carry the convergence
        dict(name="stiff_axi_256x512_mixed", kind="solve", geom="axi", n0=256, n1=512, n2=1, bubbles=1,
             precision="mixed", stiff=True, tuned=True),
        # the bubble grids of one time step in one batch, uneven sizes in multiples of 32
        dict(name="batch_24_mixed", kind="batch", count=24, lo=64, hi=1024, mixseed=5, precision="mixed"),
        # the explicit steps around the solve (coefficients, velocity and energy update) on a ragged grid
        dict(name="update_1000x616_fp64", kind="update", n0=1000, n1=616, bubbles=8),
        # the momentum predictor at the time step's dt
        dict(name="predictor_1024_fp64", kind="predictor", n0=1024, n1=1024, bubbles=16, dt=1e-7),
        # a base grid with one refined patch around the bubble
        dict(name="patch_512_fp64", kind="patch", n=512, radius=0.1, cycles=3, precision="fp64"),
    ]


def _coarsest(n, dim):
    n = list(n)
    while all(n[a] % 2 == 0 and n[a] // 2 >= 4 for a in range(dim)):
        n = [n[a] // 2 if a < dim else 1 for a in range(3)]
    return n


def _served(n):
    """2D sizes whose coarsest grid is at most 31 x 31 cells, as those of the batch and the serving loop."""
    return max(_coarsest(n, 2)) <= 31


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "solve3d", "stiff", "batch", "update", "predictor", "patch"])
    precision = rng.choice(["fp64", "mixed"])
    if kind in ("solve", "stiff"):
        while True:
            step = rng.choice([8, 16, 32, 32, 64])
            hi = 1024 if kind == "solve" else 512
            n0, n1 = (max(64, int(round(_log(rng, 64, hi) / step)) * step) for _ in range(2))
            if _served((n0, n1, 1)):
                break
        return dict(kind="solve", geom=rng.choice(["plane", "plane", "axi", "open"]), n0=n0, n1=n1, n2=1,
                    bubbles=rng.randint(1, 16) if kind == "solve" else 1, precision=precision,
                    stiff=kind == "stiff", tuned=rng.random() < 0.3)
    if kind == "solve3d":
        scale = rng.choice([8, 16, 16, 32])                   # coarsest grids of 4 to 7 cells a side
        n0, n1, n2 = (scale * rng.randint(4, 7) for _ in range(3))
        return dict(kind="solve", geom="wall3d", n0=n0, n1=n1, n2=n2, bubbles=1, precision=precision, stiff=False,
                    tuned=False)
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(4, 32), lo=64, hi=rng.choice([256, 512, 1024]),
                    mixseed=rng.randrange(1 << 20), precision=precision)
    if kind == "update":
        return dict(kind="update", n0=int(_log(rng, 40, 2000)), n1=int(_log(rng, 40, 2000)), bubbles=rng.randint(1, 16))
    if kind == "predictor":
        n0, n1 = (max(64, int(round(_log(rng, 64, 1024) / 32)) * 32) for _ in range(2))
        return dict(kind="predictor", n0=n0, n1=n1, bubbles=rng.randint(1, 16), dt=10.0 ** rng.uniform(-7, -3))
    return dict(kind="patch", n=rng.choice([64, 128, 192, 256, 384, 512]), radius=round(rng.uniform(0.05, 0.2), 3),
                cycles=rng.randint(2, 6), precision=precision)


# ------------------------------------------------------------------ inputs
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _walls(dim, axis=False):
    bc = [[WALL, WALL] for _ in range(3)]
    if axis:
        bc[0][0] = AXIS
    return tuple(tuple(s) for s in bc)


def _grid(case):
    n = (case["n0"], case["n1"], case["n2"])
    length = 6.4e-3 if case["stiff"] else 1.0
    geom = case["geom"]
    h = length / (n[1] if geom == "axi" else n[0])
    far_T, far_p = ((inputs.T_INF,) * 2,) * 3, ((inputs.P_INF,) * 2,) * 3
    if geom == "wall3d":
        bc = ((DIRICHLET, DIRICHLET), (DIRICHLET, DIRICHLET), (WALL, DIRICHLET))
        return inputs.Grid(dim=3, axisym=0, n=n, h=h, bc=bc, bcT=far_T, bcp=far_p)
    if geom == "open":
        bc = ((WALL, DIRICHLET), (DIRICHLET, DIRICHLET), (WALL, WALL))
        return inputs.Grid(dim=2, axisym=0, n=n, h=h, bc=bc, bcT=far_T, bcp=far_p)
    return inputs.Grid(dim=2, axisym=int(geom == "axi"), n=n, h=h, bc=_walls(2, geom == "axi"))


def _centres(g, dev):
    ax = [(torch.arange(g.n[a], dtype=torch.float64, device=dev) + 0.5) * g.h for a in range(3)]
    return [ax[0].view(1, 1, -1), ax[1].view(1, -1, 1), ax[2].view(-1, 1, 1)]


def _bubbles(g, rng, count, rmin, rmax):
    """Seeded centres inside the domain and radii, in lengths."""
    L = [g.n[a] * g.h for a in range(g.dim)]
    s = min(L)
    out = []
    for _ in range(count):
        R = rng.uniform(rmin, rmax) * s
        c = [rng.uniform(R, v - R) for v in L]
        if g.axisym:
            c[0] = 0.0
        if g.dim == 3:
            c[2] = rng.uniform(1.2, 1.6) * R            # a bubble near the wall at z = 0
        out.append((c, R))
    return out


def _fraction(g, bubbles, dev):
    X = _centres(g, dev)
    d = torch.full((g.n[2], g.n[1], g.n[0]), 1e30, dtype=torch.float64, device=dev)
    for c, R in bubbles:
        r2 = sum((X[a] - c[a]) ** 2 for a in range(g.dim))
        d = torch.minimum(d, r2.sqrt() - R)
    return 0.5 * (1.0 + torch.tanh(d / g.h))


def _sl(a, lo, hi):
    s = [slice(None)] * 3
    s[2 - a] = slice(lo, hi)
    return tuple(s)


def _face_mean(v, a):
    """Means of the two cells, the cell's own at the boundary."""
    return torch.cat([v[_sl(a, 0, 1)], 0.5 * (v[_sl(a, 0, -1)] + v[_sl(a, 1, None)]), v[_sl(a, -1, None)]], dim=2 - a)


def _mode(g, dev):
    X, out = _centres(g, dev), 1.0
    for a in range(g.dim):
        xi = X[a] / (g.n[a] * g.h)
        lo, hi = (g.bc[a][s] == DIRICHLET for s in (0, 1))
        out = out * (torch.sin(math.pi * xi) if lo and hi else torch.cos(0.5 * math.pi * xi) if hi else
                     torch.sin(0.5 * math.pi * xi) if lo else torch.cos(math.pi * xi))
    return out


def _problem(g, bubbles, dt, seed, dev):
    """lambda, faces, right-hand side and guess of one problem (Eqs. 29-34 with div u* = 0)."""
    C = _fraction(g, bubbles, dev)
    q, a = inputs.liquid(), inputs.gas()
    avg = lambda f1, f2: C * f1 + (1.0 - C) * f2
    gen = torch.Generator(device=dev).manual_seed(seed)
    noise = lambda: 1.0 + 1e-3 * torch.randn(C.shape, generator=gen, dtype=torch.float64, device=dev)
    phi = _mode(g, dev)
    T, p = (inputs.T_INF + 10.0 * phi) * noise(), (inputs.P_INF + 1e3 * phi) * noise()
    l1 = -avg(q.rho * q.cp, a.rho * a.cp) / dt
    l2 = avg(q.beta, a.beta) * T / dt
    br = [f.gamma / f.rho_c2 - f.beta ** 2 * inputs.T_INF / (f.rho * f.cp) for f in (q, a)]
    l3 = -avg(*br) / dt ** 2
    l4 = avg(*[f.beta / (f.rho * f.cp) for f in (q, a)]) / dt
    lam = torch.stack([l1, l2, l3, l4], dim=-1).reshape(-1, 4).contiguous()
    b = torch.stack([l1 * T + l2 * p, l3 * p], dim=-1).reshape(-1, 2).contiguous()
    x0 = torch.empty_like(b)
    x0[:, 0], x0[:, 1] = inputs.T_INF, inputs.P_INF
    fa, fk = [], []
    for ax in range(g.dim):
        Cf = _face_mean(C, ax)
        fa.append((1.0 / (Cf * q.rho + (1.0 - Cf) * a.rho)).reshape(-1).contiguous())
        fk.append((Cf * q.k + (1.0 - Cf) * a.k).reshape(-1).contiguous())
    return dict(grid=g, lam=lam, fa=fa, fk=fk, b=b, x0=x0)


def _solve_inputs(case, seed, dev):
    g = _grid(case)
    rng = np.random.default_rng(seed)
    r = (0.02, 0.08) if case["bubbles"] > 1 else (0.12, 0.2)
    return _problem(g, _bubbles(g, rng, case["bubbles"], *r), 1e-5 if case["stiff"] else 1e-7, seed, dev)


def _batch_sizes(case):
    """Log-uniform sizes in multiples of 32, fixed by the case (the seed changes the fields)."""
    rng = np.random.default_rng(case["mixseed"])
    return [min(case["hi"], max(case["lo"], 32 * int(round(math.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]))) / 32))))
            for _ in range(case["count"])]


def _batch_inputs(case, seed, dev):
    rng = np.random.default_rng(seed)
    out = []
    for q, n in enumerate(_batch_sizes(case)):
        g = inputs.Grid(dim=2, axisym=0, n=(n, n, 1), h=1.0 / n, bc=_walls(2))
        out.append(_problem(g, _bubbles(g, rng, int(rng.integers(1, 9)), 0.02, 0.08), 1e-7, 1000 * seed + q, dev))
    return out


def _state(case, seed, dev):
    """An advected state: smooth T, p and u with noise, phase densities and energies of the NASG equations."""
    n0, n1 = case["n0"], case["n1"]
    g = inputs.Grid(dim=2, axisym=0, n=(n0, n1, 1), h=1.0 / n0, bc=_walls(2))
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=dev).manual_seed(seed)
    randn = lambda s: torch.randn(s, generator=gen, dtype=torch.float64, device=dev)
    C = _fraction(g, _bubbles(g, rng, case["bubbles"], 0.02, 0.08), dev)
    xs = [(torch.arange(g.n[a], dtype=torch.float64, device=dev) + 0.5) / g.n[a] for a in range(2)]

    def smooth(amp):
        f = 0.0
        for _ in range(3):
            k, ph = rng.integers(1, 4, size=2), rng.uniform(0, 2 * math.pi, size=2)
            f = f + (torch.cos(math.pi * int(k[0]) * xs[0] + ph[0]).view(1, 1, -1) *
                     torch.cos(math.pi * int(k[1]) * xs[1] + ph[1]).view(1, -1, 1)) * rng.uniform(0.3, 1.0)
        return amp * f / 3.0 * (1.0 + 1e-3 * randn(C.shape))

    T, p = inputs.T_INF + smooth(4.0), inputs.P_INF + smooth(3e3)
    u = [smooth(0.5) for _ in range(2)]
    ph = [inputs.water_phase(), inputs.air_phase()]
    r = [inputs.phase_density(T, p, f) for f in ph]
    m = [C * r[0], (1.0 - C) * r[1]]
    rho = m[0] + m[1]
    kin = 0.5 * sum(v * v for v in u)
    Ei = [c * inputs.phase_energy(p, ri, f) + mi * kin for c, ri, f, mi in zip((C, 1.0 - C), r, ph, m)]
    uf = []
    for a in range(2):
        f = _face_mean(u[a], a)
        f = f + 5e-4 * randn(f.shape)
        f[_sl(a, 0, 1)] = 0.0
        f[_sl(a, -1, None)] = 0.0
        uf.append(f.contiguous())
    kappa = 100.0 * torch.rand(C.shape, generator=gen, dtype=torch.float64, device=dev) - 50.0
    return dict(grid=g, ph=ph, dt=1e-7, sigma=0.072, C=C, m1=m[0], m2=m[1], E=Ei[0] + Ei[1], E1=Ei[0], E2=Ei[1], rho=rho,
                mu=C * ph[0].mu + (1.0 - C) * ph[1].mu, mom=[rho * v for v in u], u=u, uf=uf, kappa=kappa, p=p, T=T)


def _patch_inputs(case, seed, dev):
    n = case["n"]
    rng = np.random.default_rng(seed)
    R = case["radius"]
    bubbles = [([0.5 + rng.uniform(-0.02, 0.02), 0.5 + rng.uniform(-0.02, 0.02)], R)]
    gb = inputs.Grid(dim=2, axisym=0, n=(n, n, 1), h=1.0 / n, bc=_walls(2))
    gf = inputs.Grid(dim=2, axisym=0, n=(2 * n, 2 * n, 1), h=0.5 / n, bc=_walls(2))
    lo = max(0, int(math.floor((0.48 - R) * n)) - 1)
    hi = min(n, int(math.ceil((0.52 + R) * n)) + 1)
    base, full = _problem(gb, bubbles, 1e-7, seed, dev), _problem(gf, bubbles, 1e-7, seed + 1, dev)
    a, b = 2 * lo, 2 * hi
    cells = lambda v, k: v.reshape(2 * n, 2 * n, k)[a:b, a:b].reshape(-1, k).contiguous()
    face = lambda f: [f[0].reshape(2 * n, 2 * n + 1)[a:b, a:b + 1].reshape(-1).contiguous(),
                      f[1].reshape(2 * n + 1, 2 * n)[a:b + 1, a:b].reshape(-1).contiguous()]
    patch = dict(lam=cells(full["lam"], 4), b=cells(full["b"], 2), x0=cells(full["x0"], 2), fa=face(full["fa"]),
                 fk=face(full["fk"]))
    return base, patch, ((lo, hi), (lo, hi))


# ------------------------------------------------------------------ state and pass
def prepare(case, seed):
    dev = torch.device("cuda")
    kind = case["kind"]
    s = dict(kind=kind, case=case)
    if kind == "solve":
        p = _solve_inputs(case, seed, dev)
        s["solver"] = binding.Solver(p["grid"], precision=case["precision"], rtol=1e-10, max_cycles=200)
        if case["tuned"]:
            s["solver"].set_coeffs(p["lam"], p["fa"], p["fk"])
            TABLE.tune(s["solver"], reps=5)
        s.update(p, x=p["x0"].clone())
    elif kind == "batch":
        s["p"] = _batch_inputs(case, seed, dev)
        s["solvers"] = [binding.Solver(p["grid"], precision=case["precision"], rtol=1e-10) for p in s["p"]]
        s["batch"] = binding.Batch(s["solvers"])
        s["x"] = [p["x0"].clone() for p in s["p"]]
    elif kind == "update":
        s.update(_state(case, seed, dev))
        g = s["grid"]
        cell = lambda k=1: torch.empty((g.N, k) if k > 1 else (g.n[2], g.n[1], g.n[0]), dtype=torch.float64, device=dev)
        face = lambda: [torch.empty(g.face_shape(a), dtype=torch.float64, device=dev) for a in range(2)]
        s["out"] = dict(lam=cell(4), b=cell(2), x0=cell(2), fa=face(), fk=face())
        s.update(uf_new=face(), p1=cell(), p2=cell(), E1n=cell(), E2n=cell())
    elif kind == "predictor":
        s.update(_state(case, seed, dev))
        g = s["grid"]
        s["solver"] = binding.Momentum(g)
        s["R"] = [torch.empty_like(s["rho"]) for _ in range(2)]
        s["x"] = [torch.empty_like(s["rho"]) for _ in range(2)]
        s["uf_new"] = [torch.empty(g.face_shape(a), dtype=torch.float64, device=dev) for a in range(2)]
    else:
        s["base"], s["patch"], box = _patch_inputs(case, seed, dev)
        s["solver"] = binding.Composite(s["base"]["grid"], box, precision=case["precision"])
        s["xb"], s["xf"] = s["base"]["x0"].clone(), s["patch"]["x0"].clone()
    return s


def run(s):
    kind = s["kind"]
    if kind == "solve":
        s["solver"].set_coeffs(s["lam"], s["fa"], s["fk"])
        s["x"].copy_(s["x0"])
        s["solver"].solve(s["b"], s["x"], allow_not_converged=s["case"]["stiff"])
        return s["x"]
    if kind == "batch":
        s["batch"].set_coeffs([p["lam"] for p in s["p"]], [p["fa"] for p in s["p"]], [p["fk"] for p in s["p"]])
        for x, p in zip(s["x"], s["p"]):
            x.copy_(p["x0"])
        s["batch"].solve([p["b"] for p in s["p"]], s["x"])
        return s["x"]
    if kind == "update":
        g, o = s["grid"], s["out"]
        binding.assemble(g, s["ph"], s["dt"], s["C"], s["m1"], s["m2"], s["E"], s["mom"], s["uf"], o)
        # the solve stands between the two in a time step; its start (T, p) takes its result's place here
        binding.correct(g, s["dt"], s["sigma"], o["x0"], s["C"], s["kappa"], o["fa"], s["uf"], s["uf_new"], s["p1"], s["p2"])
        binding.energy(g, s["ph"], s["dt"], o["x0"], s["C"], s["p1"], s["p2"], s["uf_new"], s["E1"], s["E2"], s["E1n"], s["E2n"])
        return dict(o, uf=s["uf_new"], p1=s["p1"], p2=s["p2"], E1=s["E1n"], E2=s["E2n"])
    if kind == "predictor":
        g, dt = s["grid"], s["case"]["dt"]
        binding.momentum_rhs(g, dt, s["sigma"], s["mom"], s["p"], s["kappa"], s["C"], s["R"])
        s["solver"].set_coeffs(dt, s["rho"], s["mu"])
        for x, u in zip(s["x"], s["u"]):
            x.copy_(u)
        s["solver"].solve(s["R"], s["x"], rtol=1e-10, max_iters=200)
        binding.provisional(g, dt, s["rho"], s["p"], s["x"], s["uf_new"])
        return dict(R=s["R"], u=s["x"], uf=s["uf_new"])
    b, f = s["base"], s["patch"]
    s["solver"].set_coeffs(b["lam"], b["fa"], b["fk"], f["lam"], f["fa"], f["fk"])
    s["xb"].copy_(b["x0"])
    s["xf"].copy_(f["x0"])
    s["solver"].solve(b["b"], f["b"], s["xb"], s["xf"], s["case"]["cycles"], norms=False)
    return dict(base=s["xb"], patch=s["xf"])


# Per cell: a solve reads lambda (4), the right-hand side (2), the guess (2) and 2 values per face, and writes x (2);
# its least work is one set-up and one V(2,2) cycle with its norms (75 multiply-adds per cell and level, all levels).
def _solve_work(n, dim):
    N = n[0] * n[1] * n[2]
    faces = sum(N // n[a] * (n[a] + 1) for a in range(dim))
    per = (75 if dim == 2 else 105) * (4.0 / 3.0 if dim == 2 else 8.0 / 7.0) + 45
    return 80 * N + 16 * faces, 2.0 * per * N


def work(case):
    kind = case["kind"]
    if kind == "solve":
        b, f = _solve_work((case["n0"], case["n1"], case["n2"]), 3 if case["geom"] == "wall3d" else 2)
    elif kind == "batch":
        b, f = (sum(v) for v in zip(*[_solve_work((n, n, 1), 2) for n in _batch_sizes(case)]))
    elif kind == "update":
        N = case["n0"] * case["n1"]
        b, f = (160 + 96 + 88) * N, 2.0 * (150 + 20 + 85) * N
    elif kind == "predictor":
        N = case["n0"] * case["n1"]
        b, f = 8.0 * N * (5 + 2 + 2 + 2 + 2 + 2), 2.0 * (20 + 40 + 2 * 69 + 20) * N
    else:
        m = int(2 * (2 * case["radius"] + 0.04) * case["n"])
        b1, f1 = _solve_work((case["n"], case["n"], 1), 2)
        b2, f2 = _solve_work((m, m, 1), 2)
        b, f = b1 + b2, case["cycles"] * (f1 + f2)
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ in 64 bits
def _exact_solve(p):
    """Eqs. 27-28 by block-Jacobi steps on the residual, fluxes as differences, to rounding; None where slow."""
    g = p["grid"]
    shape = (g.n[2], g.n[1], g.n[0])
    dev = p["lam"].device
    l1, l2, l3, l4 = (p["lam"][:, q].reshape(shape) for q in range(4))
    bT, bp = (p["b"][:, q].reshape(shape) for q in range(2))
    T, q = (p["x0"][:, c].reshape(shape).clone() for c in range(2))
    ri = (g.r0 + (torch.arange(g.n[0], dtype=torch.float64, device=dev) + 0.5) * g.h).view(1, 1, -1)

    def weights(a):
        if g.axisym and a == 0:
            return (ri - 0.5 * g.h) / ri, (ri + 0.5 * g.h) / ri
        return 1.0, 1.0

    def laplace(c, v, bval):
        out = torch.zeros_like(v)
        for a in range(g.dim):
            cf = c[a].reshape(g.face_shape(a))
            F = torch.zeros_like(cf)
            F[_sl(a, 1, -1)] = v[_sl(a, 1, None)] - v[_sl(a, 0, -1)]
            if g.bc[a][0] == DIRICHLET:
                F[_sl(a, 0, 1)] = 2.0 * (v[_sl(a, 0, 1)] - bval[a][0])
            if g.bc[a][1] == DIRICHLET:
                F[_sl(a, -1, None)] = 2.0 * (bval[a][1] - v[_sl(a, -1, None)])
            F = F * cf / g.h ** 2
            wl, wh = weights(a)
            out += wh * F[_sl(a, 1, None)] - wl * F[_sl(a, 0, -1)]
        return out

    def diagonal(c):
        out = torch.zeros(shape, dtype=torch.float64, device=dev)
        for a in range(g.dim):
            cf = c[a].reshape(g.face_shape(a)).clone() / g.h ** 2
            cf[_sl(a, 0, 1)] *= 2.0 if g.bc[a][0] == DIRICHLET else 0.0
            cf[_sl(a, -1, None)] *= 2.0 if g.bc[a][1] == DIRICHLET else 0.0
            wl, wh = weights(a)
            out += wh * cf[_sl(a, 1, None)] + wl * cf[_sl(a, 0, -1)]
        return out

    kT, kp = diagonal(p["fk"]), diagonal(p["fa"])
    a11, a12, a21, a22 = l1 - kT, l2, -l4 * kT, l3 - kp
    det = a11 * a22 - a12 * a21
    for _ in range(300):
        LT = laplace(p["fk"], T, g.bcT)
        rT = bT - (LT + l1 * T + l2 * q)
        rp = bp - (laplace(p["fa"], q, g.bcp) + l3 * q + l4 * LT)
        dT, dq = (a22 * rT - a12 * rp) / det, (a11 * rp - a21 * rT) / det
        T, q = T + dT, q + dq
        if max(float(dT.abs().max()) / inputs.T_INF, float(dq.abs().max()) / inputs.P_INF) < 1e-15:
            return torch.stack([T, q], dim=-1).reshape(-1, 2)
    # at the rounding of the terms the updates stop falling; further off it has not converged
    if max(float(dT.abs().max()) / inputs.T_INF, float(dq.abs().max()) / inputs.P_INF) < 1e-12:
        return torch.stack([T, q], dim=-1).reshape(-1, 2)
    return None


def _cell_derivative(v, b, h):
    return torch.cat([(v[_sl(b, 1, 2)] - v[_sl(b, 0, 1)]) / h, (v[_sl(b, 2, None)] - v[_sl(b, 0, -2)]) / (2.0 * h),
                      (v[_sl(b, -1, None)] - v[_sl(b, -2, -1)]) / h], dim=2 - b)


def _inner(F, a, v):
    F[_sl(a, 1, -1)] = v
    return F


def _div(g, F):
    return sum((F[a][_sl(a, 1, None)] - F[a][_sl(a, 0, -1)]) / g.h for a in range(g.dim))


def _exact_update(s):
    """Eqs. 10, 11, 20, 23 and 29-34, then Eq. unp1, Eqs. 37-38 and Eq. 39, on a plane grid with walls."""
    g, dt, C, ph = s["grid"], s["dt"], s["C"], s["ph"]
    Cs, ms = (C, 1.0 - C), (s["m1"], s["m2"])
    rho = s["m1"] + s["m2"]
    free = [c - m * f.b for c, m, f in zip(Cs, ms, ph)]
    shift = sum(f.Gamma * f.Pi / (f.Gamma - 1.0) * fr + m * f.q for f, fr, m in zip(ph, free, ms))
    p = (s["E"] - 0.5 * sum(m * m for m in s["mom"]) / rho - shift) / sum(fr / (f.Gamma - 1.0) for f, fr in zip(ph, free))
    T = sum(fr * p + f.Pi * fr for f, fr in zip(ph, free)) / sum(m * (f.cp - f.cv) for f, m in zip(ph, ms))
    rho_cp = beta = b_over = br = 0.0
    for c, m, f in zip(Cs, ms, ph):
        g1 = (f.Gamma - 1.0) * f.cv
        bi = g1 / (g1 * T + f.b * (p + f.Pi))
        here = c > 0.0
        ri = torch.where(here, m / torch.where(here, c, torch.ones_like(c)), torch.ones_like(c))
        c2 = f.Gamma * (p + f.Pi) / (ri * (1.0 - ri * f.b))
        rho_cp, beta = rho_cp + m * f.cp, beta + c * bi
        zero = torch.zeros_like(c)
        b_over = b_over + torch.where(here, c * bi / (ri * f.cp), zero)
        br = br + torch.where(here, c * (f.cp / f.cv / (ri * c2) - bi * bi * T / (ri * f.cp)), zero)
    l1, l2, l3, l4 = -rho_cp / dt, beta * T / dt, -br / dt ** 2, b_over / dt
    o = dict(lam=torch.stack([l1, l2, l3, l4], -1).reshape(-1, 4),
             b=torch.stack([l1 * T + l2 * p, l3 * p + _div(g, s["uf"]) / dt], -1).reshape(-1, 2),
             x0=torch.stack([T, p], -1).reshape(-1, 2), fa=[1.0 / _face_mean(rho, a) for a in range(2)], fk=[])
    for a in range(2):
        Cf = _face_mean(C, a)
        o["fk"].append(Cf * ph[0].k + (1.0 - Cf) * ph[1].k)
    uf = []
    for a in range(2):
        grad = _inner(torch.zeros_like(o["fa"][a]), a, (p[_sl(a, 1, None)] - p[_sl(a, 0, -1)]) / g.h)
        uf.append(s["uf"][a] - dt * o["fa"][a] * grad)
    sk = s["sigma"] * s["kappa"]
    pi = [p + (1.0 - C) * sk, p - C * sk]
    uc = [0.5 * (uf[a][_sl(a, 0, -1)] + uf[a][_sl(a, 1, None)]) for a in range(2)]
    E = []
    for f, q, c, Ei in zip(ph, pi, Cs, (s["E1"], s["E2"])):
        F = []
        for a in range(2):
            lo, hi, b = _sl(a, 0, -1), _sl(a, 1, None), 1 - a
            un = uf[a][_sl(a, 1, -1)]
            d = _cell_derivative(uc[a], b, g.h)
            visc = 2.0 * (uc[a][hi] - uc[a][lo]) / g.h * un
            visc = visc + (0.5 * (d[lo] + d[hi]) + (uc[b][hi] - uc[b][lo]) / g.h) * 0.5 * (uc[b][lo] + uc[b][hi])
            F.append(_inner(torch.zeros_like(uf[a]), a,
                            -0.5 * (q[lo] + q[hi]) * un + f.mu * visc + f.k * (T[hi] - T[lo]) / g.h))
        E.append(Ei + dt * c * _div(g, F))
    return dict(o, uf=uf, p1=pi[0], p2=pi[1], E1=E[0], E2=E[1])


def _exact_predictor(s, dt):
    """(rho/dt) u - div(mu (grad u + grad u^T)) = R on a plane grid with free-slip walls, by Jacobi steps."""
    g, rho, mu = s["grid"], s["rho"], s["mu"]
    zero_faces = lambda a: torch.zeros(g.face_shape(a), dtype=torch.float64, device=rho.device)
    grad = lambda v, a: _inner(zero_faces(a), a, (v[_sl(a, 1, None)] - v[_sl(a, 0, -1)]) / g.h)
    centre = lambda v, a: 0.5 * (grad(v, a)[_sl(a, 0, -1)] + grad(v, a)[_sl(a, 1, None)])
    R = [s["mom"][c] / dt - centre(s["p"], c) + s["sigma"] * s["kappa"] * centre(s["C"], c) for c in range(2)]
    muf = [_face_mean(mu, a) for a in range(2)]

    def apply(u):
        out = []
        for c in range(2):
            F = []
            for a in range(2):
                lo, hi = _sl(a, 0, -1), _sl(a, 1, None)
                n = (u[c][hi] - u[c][lo]) / g.h
                if a == c:
                    f = _inner(zero_faces(a), a, 2.0 * n)
                    f[_sl(a, 0, 1)] = 4.0 * u[c][_sl(a, 0, 1)] / g.h
                    f[_sl(a, -1, None)] = -4.0 * u[c][_sl(a, -1, None)] / g.h
                else:
                    d = _cell_derivative(u[a], c, g.h)
                    f = _inner(zero_faces(a), a, n + 0.5 * (d[lo] + d[hi]))
                F.append(muf[a] * f)
            out.append(rho / dt * u[c] - _div(g, F))
        return out

    diag = []
    for c in range(2):
        d = rho / dt
        for a in range(2):
            w = muf[a] * (2.0 if a == c else 1.0) / g.h ** 2
            d = d + w[_sl(a, 0, -1)] + w[_sl(a, 1, None)]
        diag.append(d)
    u = [v.clone() for v in s["u"]]
    for _ in range(400):
        du = [(r - y) / d for r, y, d in zip(R, apply(u), diag)]
        u = [a + b for a, b in zip(u, du)]
        top = max(float(v.abs().max()) for v in du)
        if top < 1e-15:
            break
    if top > 1e-12:
        u = [None, None]
        return dict(R=R, u=u, uf=[None, None])
    uf = []
    for a in range(2):
        w = u[a] + dt / rho * centre(s["p"], a)
        uf.append(_inner(zero_faces(a), a, 0.5 * (w[_sl(a, 0, -1)] + w[_sl(a, 1, None)])))
    return dict(R=R, u=u, uf=uf)


def exact(case, seed):
    dev = _device()
    kind = case["kind"]
    if kind == "solve":
        return None if case["stiff"] else _exact_solve(_solve_inputs(case, seed, dev))
    if kind == "batch":
        return [_exact_solve(p) for p in _batch_inputs(case, seed, dev)]
    if kind == "update":
        return _exact_update(_state(case, seed, dev))
    if kind == "predictor":
        return _exact_predictor(_state(case, seed, dev), case["dt"])
    return None                       # a fixed number of steps on a refined patch: not a converged solution
