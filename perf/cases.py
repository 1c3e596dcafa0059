"""What is timed when the solver's speed is measured: the calls that a simulation makes.

Each case goes through the public binding (``ras.Problem``, ``ras.Precond``,
``ras.BatchSolver``) on seeded synthetic reservoirs of the kind that the tests and
the benchmark use: log-normal or channelised permeability, methane, corner wells,
pressures of 1 to 10 atm, time steps of 0.1 day. ``prepare`` builds what a
simulator holds in memory between calls (handles, operators, states); ``run`` is
one pass through the entry point; ``exact`` is the same value in plain torch FP64
where the call has one (an iteration stopped at a tolerance has none).
"""
import math

import torch

from paper_2007_13966_gb300 import ras
from paper_2007_13966_gb300 import synthetic as syn

ATM, MD, DAY = 101325.0, 9.869233e-16, 86400.0
# methane, as the workloads define it
TC, PC, OMEGA, TEMP, RGAS, MOLAR, MU = 190.6, 4.599e6, 0.011, 298.0, 8.3147295, 16e-3, 11.067e-6
DT = 0.1 * DAY


def _case(kind, nx, ny, nz, **more):
    c = dict(kind=kind, nx=nx, ny=ny, nz=nz, sigma=1.0 if nz == 1 else 1.5, box=16, overlap=2, prec=32, levels=1,
             order=2, gravity=0.0, upwind=False, conservative=False, channels=False, count=1, hi=0)
    c.update(more)
    return c


def listed():
    return [
        # residual and Jacobian on the small 2D grid: the smallest call, launches count
        _case("residual", 64, 64, 1, name="residual 64x64"),
        # the same on the million-cell grid, once per Newton iteration and line-search trial
        _case("residual", 128, 128, 64, name="residual 128x128x64"),
        # Jacobian product on the layered geometry, odd sizes: once per Krylov iteration
        _case("matvec", 60, 220, 85, channels=True, name="matvec 60x220x85"),
        # the one-level preconditioner of the million-cell workload with FP32 factors
        _case("apply", 128, 128, 64, name="apply fp32 128x128x64"),
        # new factors of a new Jacobian and their first use: FP64 on the layered geometry
        _case("factor", 60, 220, 85, channels=True, prec=64, name="factor fp64 60x220x85"),
        # the same with BF16-stored factors on a ragged grid (boxes of several shapes)
        _case("factor", 97, 61, 33, overlap=1, prec=16, name="factor bf16 97x61x33"),
        # the 2D workload's linear solve: FP64, 4x4 subdomains, every call short
        _case("gmres", 64, 64, 1, overlap=1, prec=64, order=1, name="gmres fp64 64x64"),
        # one implicit step of the million-cell workload, two-level V-cycle, FP32 factors
        _case("newton", 128, 128, 64, levels=2, name="step fp32 128x128x64"),
        # the all-FP64 form of an implicit step, as used for reference runs
        _case("newton", 64, 64, 32, levels=2, prec=64, name="step fp64 64x64x32"),
        # one implicit step of the layered workload with the three-level V-cycle
        _case("newton", 60, 220, 85, levels=3, channels=True, name="step 3 levels 60x220x85"),
        # one step of a batch of independent reservoirs of uneven sizes
        _case("batch", 32, 32, 32, levels=2, overlap=1, count=12, hi=64, name="batch of 12, 32 to 64"),
        # one step of the adjoint's backward loop: transposed Jacobian, right-RAS, FGMRES, gradient
        _case("adjoint", 128, 128, 32, levels=2, prec=64, name="adjoint 128x128x32"),
    ]


def _edges(rng, cells, flat):
    """Edges of a grid of about `cells` cells, some of them odd, aspect ratios up to 3."""
    d = 2 if flat else 3
    w = [rng.uniform(-0.5, 0.5) for _ in range(d)]
    e = [max(8, int(round(math.exp(math.log(cells) / d + v - sum(w) / d)))) for v in w]
    return (e[0], e[1], 1) if flat else tuple(e)


def draw(rng):
    kind = rng.choice(["residual", "residual", "matvec", "apply", "apply", "factor", "factor", "gmres", "newton",
                       "newton3", "batch", "adjoint"])
    lo, hi = {"residual": (4e3, 1.1e6), "matvec": (4e3, 1.1e6), "apply": (4e3, 1.1e6), "factor": (4e3, 1.1e6),
              "gmres": (4e3, 1.2e5), "newton": (3e4, 6e5), "newton3": (3e4, 4e5), "batch": (3e4, 6e4),
              "adjoint": (3e4, 4e5)}[kind]
    cells = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    flat = kind in ("residual", "matvec", "apply", "factor", "gmres") and cells < 1e5 and rng.random() < 0.4
    nx, ny, nz = _edges(rng, cells, flat)
    more = dict(sigma=round(rng.uniform(0.5, 1.5), 3), box=rng.randint(12, 20), overlap=rng.randint(1, 2))
    if kind == "residual":
        more.update(order=rng.randint(1, 2), gravity=rng.choice([0.0, 0.0, 9.81]), upwind=rng.random() < 0.25,
                    conservative=rng.random() < 0.25)
    elif kind in ("apply", "factor"):
        more.update(prec=rng.choice([64, 32, 32, 16]))
    elif kind == "gmres":
        more.update(prec=rng.choice([64, 32]), order=1)
    elif kind == "newton":
        more.update(levels=2, prec=rng.choice([64, 32, 32]))
        if more["prec"] == 64:
            nx, ny, nz = _edges(rng, min(cells, 1.5e5), False)
    elif kind == "newton3":
        kind = "newton"
        more.update(levels=3, channels=rng.random() < 0.5)
    elif kind == "batch":
        more.update(levels=2, count=rng.randint(3, 10), hi=rng.randint(40, 60), overlap=1)
        nx = ny = nz = rng.randint(24, 36)
    elif kind == "adjoint":
        more.update(levels=2, prec=64)
    return _case(kind, nx, ny, nz, **more)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _rng(seed, stream):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + stream) % (1 << 62))


def _smooth(shape, corr, gen):
    """Unit-variance Gaussian field on the grid [nz, ny, nx], correlated over `corr` cells."""
    f = torch.randn(shape, generator=gen, dtype=torch.float64, device="cuda")
    for ax, n in enumerate(shape):
        if n > 1:
            x = torch.arange(n, dtype=torch.float64, device="cuda")
            W = torch.exp(-0.5 * ((x[:, None] - x[None, :]) / corr) ** 2)
            W /= W.sum(1, keepdim=True)
            f = torch.movedim(torch.tensordot(W, f, dims=([1], [ax])), 0, ax)
    return (f - f.mean()) / f.std()


def _rock(case, seed, dims):
    """Permeability and porosity [N] on the device, and the cell sizes."""
    nx, ny, nz = dims
    if case["channels"]:
        r = syn.channelised_reservoir(nx, ny, nz, seed_k=int(seed) % (1 << 31), seed_phi=(int(seed) + 1) % (1 << 31))
        g = r.grid
        return (torch.as_tensor(r.kx, device="cuda"), torch.as_tensor(r.phi, device="cuda"), (g.hx, g.hy, g.hz))
    gen = _rng(seed, 1)
    k = (100.0 * MD * torch.exp(case["sigma"] * _smooth((nz, ny, nx), 8.0, gen))).reshape(-1)
    phi = 0.15 + 0.1 * torch.rand(nx * ny * nz, generator=gen, dtype=torch.float64, device="cuda")
    h = (100.0 / 64, 100.0 / 64, 1.0) if nz == 1 else (100.0 / 128, 100.0 / 128, 50.0 / 64)
    return k, phi, h


def _reservoir(case, seed, dims=None):
    nx, ny, nz = dims or (case["nx"], case["ny"], case["nz"])
    k, phi, h = _rock(case, seed, (nx, ny, nz))
    grid = syn.Grid(nx, ny, nz, *h)
    kh = k.cpu().numpy()
    return syn.Reservoir(grid, syn.Fluid(), kh, kh, kh, phi.cpu().numpy(), syn.corner_wells(grid, kh), dt=DT,
                         gravity=case["gravity"], upwind=case["upwind"], conservative=case["conservative"])


def _states(case, seed):
    """Three time levels of a smooth pressure field between 1 and 10 atm."""
    shape = (case["nz"], case["ny"], case["nx"])
    gen = _rng(seed, 2)
    u = 0.5 * (1.0 + torch.tanh(_smooth(shape, 3.0, gen)))
    p = ((1.0 + 9.0 * u) * ATM).reshape(-1)
    v = (1.0 + 0.01 * _smooth(shape, 3.0, gen)).reshape(-1)
    return p.contiguous(), (p * v).contiguous(), (p * v * v).contiguous()


def _vector(case, seed, stream):
    return torch.randn(case["nx"] * case["ny"] * case["nz"], generator=_rng(seed, stream), dtype=torch.float64,
                       device="cuda")


def _parts(case, dims=None):
    return tuple(-(-n // case["box"]) for n in (dims or (case["nx"], case["ny"], case["nz"])))


def _precond(case, gp, dims=None, **more):
    ratio = (2, 2, 2) if case["levels"] == 3 else (4, 4, 4)
    return ras.Precond(gp, _parts(case, dims), case["overlap"], factor_prec=case["prec"], nlevels=case["levels"],
                       coarsen=ratio, coarse_prec=64 if case["prec"] == 64 else 32, **more)


def _operator(case, seed, s):
    """Problem handle and the Jacobian at a smooth state."""
    s["gp"] = ras.Problem(_reservoir(case, seed))
    s["p"], s["pl"], s["plm1"] = _states(case, seed)
    s["F"] = torch.zeros_like(s["p"])
    s["gp"].residual_eval(s["p"], s["pl"], s["plm1"], DT, case["order"], s["F"], s["gp"].J)


def prepare(case, seed):
    kind, s = case["kind"], {"case": case}
    if kind in ("residual", "matvec", "apply", "factor"):
        _operator(case, seed, s)
        s["r"] = _vector(case, seed, 3)
        s["z"] = torch.zeros_like(s["r"])
        if kind in ("apply", "factor"):
            s["pc"] = _precond(case, s["gp"])
            s["pc"].factor(s["gp"].J)
    elif kind == "gmres":
        # the first Newton system of a simulation that starts from rest
        s["gp"] = ras.Problem(_reservoir(case, seed))
        p = torch.full((s["gp"].N,), ATM, dtype=torch.float64, device="cuda")
        F = torch.zeros_like(p)
        s["gp"].residual_eval(p, p, None, DT, 1, F, s["gp"].J)
        s["b"], s["x"] = -F, torch.zeros_like(F)
        s["pc"] = _precond(case, s["gp"])
        s["pc"].factor(s["gp"].J)
    elif kind == "newton":
        # the second implicit step (BDF2) of a simulation that starts from rest
        s["gp"] = ras.Problem(_reservoir(case, seed))
        s["pc"] = _precond(case, s["gp"])
        s["plm1"] = torch.full((s["gp"].N,), ATM, dtype=torch.float64, device="cuda")
        s["pl"] = s["plm1"].clone()
        s["gp"].newton_step(s["pc"], s["pl"], s["plm1"], None, DT, 1)
    elif kind == "batch":
        r = torch.Generator().manual_seed(case["count"] * 7919 + case["nx"] * 104729 + case["hi"])
        edges = torch.randint(case["nx"], case["hi"] + 1, (case["count"],), generator=r).tolist()
        s["gps"], s["pcs"] = [], []
        for i, n in enumerate(edges):
            s["gps"].append(ras.Problem(_reservoir(case, seed * 64 + i, (n, n, n))))
            s["pcs"].append(_precond(case, s["gps"][-1], (n, n, n)))
        s["solver"] = ras.BatchSolver(s["gps"], s["pcs"])
        s["plm1"] = [torch.full((g.N,), ATM, dtype=torch.float64, device="cuda") for g in s["gps"]]
        s["pl"] = [q.clone() for q in s["plm1"]]
        s["solver"].newton_step(s["pl"], s["plm1"], None, [DT] * len(edges), 1)
    elif kind == "adjoint":
        s["gp"] = ras.Problem(_reservoir(case, seed))
        s["p"], s["pl"], s["plm1"] = _states(case, seed)
        N = s["gp"].N
        z = lambda: torch.zeros(N, dtype=torch.float64, device="cuda")
        s["F"], s["rhs"], s["dphi"], s["x"], s["grad"] = z(), z(), z(), z(), z()
        s["JT"] = [z() for _ in range(7)]
        s["lam1"], s["lam2"] = _vector(case, seed, 4), _vector(case, seed, 5)
        s["dphi"][N - 1] = 2.0 * s["p"][N - 1]
        s["pc"] = _precond(case, s["gp"], ras_type=2)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "residual":
        s["gp"].residual_eval(s["p"], s["pl"], s["plm1"], DT, case["order"], s["F"], s["gp"].J)
        return [s["F"]] + s["gp"].J
    if kind == "matvec":
        s["gp"].matvec(s["gp"].J, s["r"], s["z"])
        return s["z"]
    if kind == "apply":
        s["pc"].apply(s["r"], s["z"])
        return s["z"]
    if kind == "factor":
        s["pc"].factor(s["gp"].J)
        s["pc"].apply(s["r"], s["z"])
        return s["z"]
    if kind == "gmres":
        s["gp"].gmres_solve(s["gp"].J, s["pc"], s["b"], s["x"], restart=30, rtol=1e-6)
        return s["x"]
    if kind == "newton":
        p = s["pl"].clone()
        s["gp"].newton_step(s["pc"], p, s["pl"], s["plm1"], DT, 2)
        return p
    if kind == "batch":
        ps = [q.clone() for q in s["pl"]]
        s["solver"].newton_step(ps, s["pl"], s["plm1"], [DT] * len(ps), 2)
        return ps
    # adjoint: J at the checkpointed state, its transpose, the right-hand side with the
    # two later levels, the transposed solve, this level's part of the gradient
    gp = s["gp"]
    gp.residual_eval(s["p"], s["pl"], s["plm1"], DT, 2, s["F"], gp.J)
    gp.stencil_transpose(gp.J, s["JT"])
    gp.adjoint_rhs(s["dphi"], s["pl"], s["lam1"], 2.0 / DT, s["plm1"], s["lam2"], -0.5 / DT, s["rhs"])
    s["pc"].factor(s["JT"])
    gp.gmres_solve(s["JT"], s["pc"], s["rhs"], s["x"], restart=30, rtol=1e-12)
    s["grad"].zero_()
    gp.grad_logk(s["p"], s["x"], s["grad"])
    return [s["rhs"], s["x"], s["grad"]]


def _box_cells(case, dims):
    """Cells of all overlapped boxes."""
    total = 1
    for n, parts in zip(dims, _parts(case, dims)):
        total *= sum(hi - lo for lo, hi in _boxes(n, parts, case["overlap"]))
    return total


def work(case):
    """Each input read once, each output written once, per operation of the method.
    A step is counted with 3 Newton iterations of 9 Krylov iterations each."""
    dims = (case["nx"], case["ny"], case["nz"])
    n, kind, val = dims[0] * dims[1] * dims[2], case["kind"], case["prec"] / 8.0
    if kind == "batch":
        r = torch.Generator().manual_seed(case["count"] * 7919 + case["nx"] * 104729 + case["hi"])
        edges = torch.randint(case["nx"], case["hi"] + 1, (case["count"],), generator=r).tolist()
        n = sum(e ** 3 for e in edges)
        boxes = sum(_box_cells(case, (e, e, e)) for e in edges)
    else:
        boxes = _box_cells(case, dims)
    resid = {"bytes": 120.0 * n, "flops": 160.0 * n}          # p at three levels, phi, T; F and 7 arrays
    matvec = {"bytes": 72.0 * n, "flops": 13.0 * n}
    apply = {"bytes": 7.0 * val * boxes + 16.0 * n, "flops": 13.0 * boxes}
    factor = {"bytes": 56.0 * n + 7.0 * val * boxes, "flops": 10.0 * boxes}
    parts = {"residual": [(1, resid)], "matvec": [(1, matvec)], "apply": [(1, apply)],
             "factor": [(1, factor), (1, apply)]}.get(kind)
    if parts is None:
        smooth = 1 if case["levels"] == 1 else 2
        its = 9 if case["levels"] > 1 else 40
        ortho = {"bytes": 8.0 * n * (its + 4), "flops": 8.0 * n * its}
        krylov = [(its, matvec), (its * smooth, apply), (its, ortho)]
        if kind == "gmres":
            parts = krylov
        elif kind == "adjoint":
            parts = [(1, resid), (1, factor)] + [(2 * k, w) for k, w in krylov] + [(1, {"bytes": 200.0 * n, "flops": 200.0 * n})]
        else:
            parts = [(4, resid), (3, factor)] + [(3 * k, w) for k, w in krylov]
    return {m: float(sum(k * w[m] for k, w in parts)) for m in ("bytes", "flops")}


# ---------------------------------------------------------------------------
# exact values in plain torch FP64
# ---------------------------------------------------------------------------

def _pr_constants():
    m = 0.37464 + 1.54226 * OMEGA - 0.26992 * OMEGA ** 2
    a = 0.45724 * (RGAS * TC) ** 2 / PC * (1.0 + m * (1.0 - math.sqrt(TEMP / TC))) ** 2
    return a / (RGAS * TEMP) ** 2, 0.0778 * RGAS * TC / PC / (RGAS * TEMP)


def _gas(p):
    """Z, c = d(p/Z)/dp, dc/dp, m = p/(mu Z), dm/dp of the Peng-Robinson gas (one real root here)."""
    al, be = _pr_constants()
    A, B = al * p, be * p
    Z = torch.ones_like(p)
    for _ in range(12):
        f = Z ** 3 - (1 - B) * Z ** 2 + (A - 3 * B ** 2 - 2 * B) * Z - (A * B - B ** 2 - B ** 3)
        Z = Z - f / (3 * Z ** 2 - 2 * (1 - B) * Z + (A - 3 * B ** 2 - 2 * B))
    fZ = 3 * Z ** 2 - 2 * (1 - B) * Z + (A - 3 * B ** 2 - 2 * B)
    fp = be * Z ** 2 + (al - 6 * be * B - 2 * be) * Z - (2 * al * B - 2 * be * B - 3 * be * B ** 2)
    dZ = -fp / fZ
    fZZ, fZp = 6 * Z - 2 * (1 - B), 2 * be * Z + al - 6 * be * B - 2 * be
    fpp = -6 * be ** 2 * Z - (2 * al * be - 2 * be ** 2 - 6 * be ** 2 * B)
    d2Z = -(fZZ * dZ ** 2 + 2 * fZp * dZ + fpp) / fZ
    c = 1 / Z - p * dZ / Z ** 2
    dc = -2 * dZ / Z ** 2 - p * d2Z / Z ** 2 + 2 * p * dZ ** 2 / Z ** 3
    return Z, c, dc, p / (MU * Z), c / MU


def _exact_residual(case, seed):
    """F and the seven arrays of its Jacobian, [nz, ny, nx] each."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    k, phi, h = _rock(case, seed, (nx, ny, nz))
    k, phi = k.reshape(nz, ny, nx), phi.reshape(nz, ny, nx)
    p, pl, plm1 = (q.reshape(nz, ny, nx) for q in _states(case, seed))
    vol = h[0] * h[1] * h[2]
    Z, c, dc, m, dm = _gas(p)
    one = case["order"] == 1
    rate = (lambda a, b, d: (a - b) / DT) if one else (lambda a, b, d: (3 * a - 4 * b + d) / (2 * DT))
    w = (1.0 if one else 1.5) / DT
    if case["conservative"]:
        F, J0 = vol * phi * rate(p / Z, pl / _gas(pl)[0], plm1 / _gas(plm1)[0]), vol * phi * c * w
    else:
        D = rate(p, pl, plm1)
        F, J0 = vol * phi * c * D, vol * phi * (dc * D + c * w)
    J = [J0] + [torch.zeros_like(p) for _ in range(6)]
    ghz = case["gravity"] * h[2] * MOLAR * MU / (RGAS * TEMP)
    for ax, slot, area, d in ((2, 1, h[1] * h[2], h[0]), (1, 3, h[0] * h[2], h[1]), (0, 5, h[0] * h[1], h[2])):
        n = p.shape[ax]
        if n < 2:
            continue
        a = lambda t: t.narrow(ax, 0, n - 1)
        b = lambda t: t.narrow(ax, 1, n - 1)
        T = area / (d / (2 * a(k)) + d / (2 * b(k)))
        g = ghz if ax == 0 else 0.0
        mean = 0.5 * (a(m) + b(m))
        dphi = (a(p) - b(p)) + g * mean          # the second cell is the deeper one
        wa = torch.where(dphi >= 0, 1.0, 0.0) if case["upwind"] else torch.full_like(dphi, 0.5)
        mf = wa * a(m) + (1 - wa) * b(m)
        flux = T * mf * dphi
        da = T * (wa * a(dm) * dphi + mf * (1 + 0.5 * g * a(dm)))
        db = T * ((1 - wa) * b(dm) * dphi + mf * (-1 + 0.5 * g * b(dm)))
        a(F).add_(flux)
        b(F).sub_(flux)
        a(J[0]).add_(da)
        b(J[0]).sub_(db)
        a(J[slot + 1]).copy_(db)
        b(J[slot]).copy_(-da)
    for at, pw in (((slice(None), 0, 0), 10 * ATM), ((slice(None), ny - 1, nx - 1), ATM)):
        T = 2.0 * k[at] * h[1] * h[2] / h[0]
        mw = _gas(torch.full_like(p[at], pw))[3]
        dp = p[at] - pw
        wa = torch.where(dp >= 0, 1.0, 0.0) if case["upwind"] else torch.full_like(dp, 0.5)
        mf = wa * m[at] + (1 - wa) * mw
        F[at] += T * mf * dp
        J[0][at] += T * (wa * dm[at] * dp + mf)
    return F, J


def _boxes(n, parts, overlap):
    cut = [q * (n // parts) + min(q, n % parts) for q in range(parts + 1)]
    return [(max(cut[q] - overlap, 0), min(cut[q + 1] + overlap, n)) for q in range(parts)]


def _exact_apply(case, J, r):
    """Left-RAS: ILU(0) solves in every overlapped box, each cell from its owning box."""
    dims = (case["nx"], case["ny"], case["nz"])
    nx, ny, nz = dims
    parts = _parts(case)
    spans = [_boxes(n, q, case["overlap"]) for n, q in zip(dims, parts)]
    cuts = [[q * (n // k) + min(q, n % k) for q in range(k + 1)] for n, k in zip(dims, parts)]
    shapes = {}
    for kz in range(parts[2]):
        for jy in range(parts[1]):
            for ix in range(parts[0]):
                e = [spans[a][q] for a, q in enumerate((ix, jy, kz))]
                shapes.setdefault(tuple(hi - lo for lo, hi in e), []).append(((ix, jy, kz), [lo for lo, _ in e]))
    C = [j.reshape(-1) for j in J]
    z = torch.zeros_like(r)
    for (bx, by, bz), boxes in shapes.items():
        i, j, k = (torch.arange(b, device=r.device) for b in (bx, by, bz))
        K, Jj, I = torch.meshgrid(k, j, i, indexing="ij")
        K, Jj, I = K.reshape(-1), Jj.reshape(-1), I.reshape(-1)
        off = torch.tensor([o[0] + nx * (o[1] + ny * o[2]) for _, o in boxes], device=r.device)
        cell = (I + nx * (Jj + ny * K))[:, None] + off[None, :]          # [box cells, boxes]
        n, dist = bx * by * bz, (1, bx, bx * by)
        low = [C[s][cell] for s in (1, 3, 5)]
        up = [C[s][cell] for s in (2, 4, 6)]
        for ax, (q, b) in enumerate(((I, bx), (Jj, by), (K, bz))):
            low[ax][q == 0] = 0.0
            up[ax][q == b - 1] = 0.0
        order = torch.argsort(I + Jj + K, stable=True)
        width = torch.bincount(I + Jj + K).tolist()
        levels = list(torch.split(order, width))
        prev = [[(lv - d).clamp_(min=0) for d in dist] for lv in levels]  # outside: a zero coefficient
        nxt = [[(lv + d).clamp_(max=n - 1) for d in dist] for lv in levels]
        D, y = C[0][cell], r[cell]
        for q, (lv, pv) in enumerate(zip(levels, prev)):
            d, t = D[lv], y[lv]
            for a in (2, 1, 0) if q else ():
                d = d - low[a][lv] / D[pv[a]] * up[a][pv[a]]
                t = t - low[a][lv] * y[pv[a]]
            D[lv] = d
            y[lv] = t / d
        for q in range(len(levels) - 2, -1, -1):
            lv = levels[q]
            y[lv] = y[lv] - sum(up[a][lv] * y[nxt[q][a]] for a in range(3)) / D[lv]
        for b, ((ix, jy, kz), o) in enumerate(boxes):
            own = torch.ones(n, dtype=torch.bool, device=r.device)
            for q, a, t in ((I, 0, ix), (Jj, 1, jy), (K, 2, kz)):
                own &= (q + o[a] >= cuts[a][t]) & (q + o[a] < cuts[a][t + 1])
            z[cell[own, b]] = y[own, b]
    return z


def exact(case, seed):
    if case["kind"] not in ("residual", "matvec", "apply", "factor"):
        return None      # iterations stopped at a tolerance: no closed value
    F, J = _exact_residual(case, seed)
    if case["kind"] == "residual":
        return [F.reshape(-1)] + [j.reshape(-1) for j in J]
    r = _vector(case, seed, 3)
    if case["kind"] != "matvec":
        return _exact_apply(case, J, r)
    x = r.reshape(J[0].shape)
    y = J[0] * x
    for ax, slot in ((2, 1), (1, 3), (0, 5)):
        n = x.shape[ax]
        y.narrow(ax, 1, n - 1).add_(J[slot].narrow(ax, 1, n - 1) * x.narrow(ax, 0, n - 1))
        y.narrow(ax, 0, n - 1).add_(J[slot + 1].narrow(ax, 0, n - 1) * x.narrow(ax, 1, n - 1))
    return y.reshape(-1)
