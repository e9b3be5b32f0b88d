"""The work that a user of this framework has it do, as cases that can be timed and compared.

A case names one call (or one step made of calls) of the public API, its grid and its options:

* ``solve``     Context.solve on a context already built: one pressure solve;
* ``project``   one time step's projection: face_coeffs, Context.update, Context.project
                (``grid="stretched"``: with stretched_metrics; ``grid="cut"``: fractional face areas);
* ``gradient``  autograd.project and its backward: one step of a training or control loop;
* ``step``      Context.rk2_step: a whole Runge-Kutta time step (two projections, momentum, VOF);
* ``momentum``  momentum_rhs alone, which takes any grid.

Sizes come from the repository's workloads (32^3, 64^3, 128^3 and 256^3 cubes, the 512x256x128 tank,
the 1024x512x256 wave, the stretched and cut-cell variants) and its ragged test grids.
"""
import math
import random

import torch

from paper_1410_2240_gb300 import autograd, mgproj

RHO_AIR, RHO_WATER = 1.0e-3, 1.0   # density ratio of air and water
TOL = 1.0e-10                      # the API's default tolerance
FORCES = dict(g=1.0, inv_re=1.0e-6, mu_air=1.8e-2, mu_water=1.0, convection=True)


def listed():
    def case(name, kind, nx, ny, nz, precision="mixed", surface="waves", body=True, grid="uniform"):
        return dict(name=name, kind=kind, nx=nx, ny=ny, nz=nz, precision=precision, surface=surface, body=body,
                    grid=grid)
    return [
        # the smallest workload, library defaults (plain FP64 cycles): launches and latency count
        case("solve_fp64_32", "solve", 32, 32, 32, "fp64", body=False),
        # the 128^3 workload with a body, library defaults
        case("solve_fp64_128", "solve", 128, 128, 128, "fp64"),
        # a small training step at autograd.project's default precision
        case("gradient_fp64_64", "gradient", 64, 64, 64, "fp64"),
        # a time step's projection on a coarse grid whose spacing is not a power of two
        case("project_mixed_96", "project", 96, 96, 96),
        # an ordinary training step
        case("gradient_mixed_128", "gradient", 128, 128, 128),
        # a ragged grid stretched along z, as the paper's runs stretch theirs
        case("project_stretched", "project", 192, 160, 224, grid="stretched"),
        # the benchmark's step, in both precisions
        case("gradient_mixed_256", "gradient", 256, 256, 256),
        case("gradient_fp64_256", "gradient", 256, 256, 256, "fp64"),
        # the towing tank with entrained air
        case("gradient_mixed_tank", "gradient", 512, 256, 128, surface="bubbles", body=False),
        # the largest grid: a plunging wave and a hull
        case("project_mixed_1024", "project", 1024, 512, 256, surface="plunging"),
        # a whole time step of the solver
        case("step_mixed_256", "step", 256, 256, 256),
        # the momentum terms alone, on a grid of odd sizes that no multigrid hierarchy takes
        case("momentum_ragged", "momentum", 251, 190, 133, "fp64"),
    ]


def draw(rng: random.Random):
    """One more case: a call of `listed`'s kinds on a grid of up to 2^24 cells."""
    kind = rng.choice(["solve", "project", "project", "gradient", "gradient", "step", "momentum"])
    cells = 2.0 ** rng.uniform(12.5, 24.0)
    if kind == "momentum":
        n = cells ** (1.0 / 3.0)
        nx, ny = (max(8, round(n * 2.0 ** rng.uniform(-0.7, 0.7))) for _ in range(2))
        nz = max(8, min(int(2 ** 24 / (nx * ny)), round(cells / (nx * ny))))
    else:
        while True:  # a coarsest grid of at most 512 cells, doubled along every axis
            a = [rng.choice([4, 4, 5, 6, 7, 8, 9, 12, 16]) for _ in range(3)]
            k = max(1, round(math.log2(cells / (a[0] * a[1] * a[2])) / 3.0))
            nx, ny, nz = (v << k for v in a)
            if a[0] * a[1] * a[2] <= 512 and 4096 <= nx * ny * nz <= 2 ** 24:
                break
    grid = rng.choice(["uniform", "uniform", "stretched", "cut"]) if kind == "project" else "uniform"
    return dict(kind=kind, nx=nx, ny=ny, nz=nz, precision="fp64" if kind == "momentum" else rng.choice(["mixed", "fp64"]),
                surface=rng.choice(["waves", "bubbles", "plunging"]), body=grid == "uniform" and rng.random() < 0.6,
                grid=grid)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _geometry(case, seed):
    """phi (the water's volume fraction), the solid mask or None and h, on a box of height 1."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    h = 1.0 / nz
    r = random.Random(seed)
    ax = [(torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * h for n in (nx, ny, nz)]
    x, y, z = ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]
    lx, ly = nx * h, ny * h
    profile = lambda s: 0.5 * (1.0 - torch.tanh(s / (1.5 * h)))
    if case["surface"] == "plunging":  # an overturned crest
        zeta = z - 0.5
        xi = (x - 0.6 * lx - 40.0 * zeta ** 3) / min(0.12, 0.1 * lx)
        crest = 0.15 * (1.0 + 0.2 * torch.cos(math.pi * y / ly + r.uniform(0.0, 2.0 * math.pi)))
        phi = profile(zeta - crest * torch.exp(-xi ** 2))
    else:  # four random modes, of the height of waves or of ripples
        s = sum(torch.cos(2.0 * math.pi * (m * x / lx + r.randint(-m, m) * y / ly) + r.uniform(0.0, 2.0 * math.pi))
                for m in range(1, 5))
        amp = 0.08 if case["surface"] == "waves" else 0.01
        phi = profile(z - 0.5 - amp * s / s.abs().max())
    if case["surface"] == "bubbles":  # air bubbles of radius 2 to 6 cells under the surface
        for _ in range(max(4, nx * ny * nz // 84000)):
            rad = r.uniform(2.0, 6.0) * h
            c = [r.uniform(0.0, lx), r.uniform(0.0, ly), r.uniform(0.0, 0.45)]
            w = rad + 12.0 * h
            lo = [max(0, int((v - w) / h)) for v in c]
            hi = [min(n, int((v + w) / h) + 1) for v, n in zip(c, (nx, ny, nz))]
            d = torch.sqrt((ax[0][lo[0]:hi[0]] - c[0])[None, None, :] ** 2 + (ax[1][lo[1]:hi[1]] - c[1])[None, :, None] ** 2
                           + (ax[2][lo[2]:hi[2]] - c[2])[:, None, None] ** 2)
            box = phi[lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]]
            torch.minimum(box, profile(rad - d), out=box)
    solid = None
    if case["body"]:  # a body that pierces the surface
        q = ((x / lx - 0.5) / 0.3) ** 2 + ((y / ly - 0.5) / 0.12) ** 2 + ((z - 0.5) / 0.1) ** 2
        solid = (q <= 1.0).to(torch.uint8)
    return phi.contiguous(), solid, h


def _open(shape, solid):
    """1 on open faces, 0 on walls and on faces that touch the body, for each axis."""
    out = []
    for a in (2, 1, 0):
        o = torch.ones(shape, dtype=torch.float64, device="cuda")
        o.narrow(a, 0, 1).zero_()
        if solid is not None:
            n = shape[a] - 1
            live = (solid == 0).to(torch.float64)
            o.mul_(live)
            o.narrow(a, 1, n).mul_(live.narrow(a, 0, n))
        out.append(o)
    return tuple(out)


def _inputs(case, seed):
    phi, solid, h = _geometry(case, seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    normal = lambda sigma: tuple(torch.randn(phi.shape, generator=gen, dtype=torch.float64, device="cuda") * sigma * o
                                 for o in _open(phi.shape, solid))
    d = dict(phi=phi, solid=solid, h=h, dt=1.0, u=normal(0.1))
    if case["kind"] == "solve":
        d["rhs"] = torch.randn(phi.shape, generator=gen, dtype=torch.float64, device="cuda")
        if solid is not None:
            d["rhs"] *= (solid == 0)
        d["rhs"] -= d["rhs"].sum() / (phi.numel() if solid is None else (solid == 0).sum())
        if solid is not None:
            d["rhs"] *= (solid == 0)
    if case["kind"] == "gradient":
        d["w"] = normal(1.0)
    if case["kind"] == "step":
        d["dt"] = 0.2 * h
    if case["grid"] == "stretched":  # widths 3.5 : 1 along z, the finest at the free surface
        t = (torch.arange(case["nz"], dtype=torch.float64, device="cuda") + 0.5) / case["nz"]
        hz = 1.0 + 2.5 * (0.5 + 0.5 * torch.cos(2.0 * math.pi * t))
        full = lambda n: torch.full((n,), h, dtype=torch.float64, device="cuda")
        d["widths"] = (full(case["nx"]), full(case["ny"]), (hz / hz.sum()).contiguous())
    if case["grid"] == "cut":  # the body as a level set at the grid's nodes
        n = [torch.arange(v + 1, dtype=torch.float64, device="cuda") / v for v in (case["nx"], case["ny"], case["nz"])]
        q = (((n[0] - 0.5) / 0.3) ** 2)[None, None, :] + (((n[1] - 0.5) / 0.12) ** 2)[None, :, None] \
            + (((n[2] - 0.5) / 0.1) ** 2)[:, None, None]
        d["psi"] = ((torch.sqrt(q) - 1.0) * 0.1).contiguous()
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    s = dict(d, kind=case["kind"], grid=case["grid"], precision=case["precision"])
    if case["kind"] == "gradient":  # autograd.project keeps its own context
        s["u"] = tuple(x.requires_grad_(True) for x in s["u"])
        s["phi"] = s["phi"].requires_grad_(True)
        return s
    s["beta"] = mgproj.face_coeffs(d["phi"], d["h"], d["solid"], RHO_AIR, RHO_WATER)
    if case["kind"] == "momentum":
        s["forces"] = mgproj.forces(**FORCES)
        s["work"] = torch.empty(12 * d["phi"].numel(), dtype=torch.float64, device="cuda")
        return s
    mixed = case["precision"] == "mixed"
    if case["kind"] == "solve":
        opts = dict(prec="mixed", krylov=1, inner_cycles=2) if mixed else {}  # {}: the library's defaults
    else:
        opts = dict(prec=case["precision"], krylov=1, inner_cycles=2 if mixed else 1)
    if case["grid"] == "stretched":
        bidx, area = mgproj.stretched_metrics(*d["widths"], s["beta"])
        s["ctx"] = mgproj.Context(bidx, 1.0, **opts)
        s["ctx"].set_face_areas(area)
    else:
        s["ctx"] = mgproj.Context(s["beta"], d["h"], **opts)
        if case["grid"] == "cut":
            s["ctx"].set_face_areas(mgproj.face_areas(d["psi"], d["h"]))
    if case["kind"] == "step":
        s["forces"] = mgproj.forces(**FORCES)
        s["now"] = tuple(torch.empty_like(x) for x in d["u"])
    return s


def run(s):
    if s["kind"] == "solve":
        return {"p": s["ctx"].solve(s["rhs"], tol=TOL)[0]}
    if s["kind"] == "gradient":
        u, p = autograd.project(s["u"], s["phi"], s["h"], solid=s["solid"], dt=s["dt"], rho_air=RHO_AIR,
                                rho_water=RHO_WATER, tol=TOL, precision=s["precision"])
        g = torch.autograd.grad(u, s["u"] + (s["phi"],), grad_outputs=s["w"])
        return {"u": tuple(x.detach() for x in u), "p": p.detach(), "grad_u": g[:3], "grad_phi": g[3]}
    if s["kind"] == "momentum":
        return {"R": mgproj.momentum_rhs(s["phi"], s["beta"], s["u"], s["h"], s["forces"], work=s["work"])}
    if s["kind"] == "step":
        for a, b in zip(s["now"], s["u"]):  # the step advances the velocity in place: from the same state each time
            a.copy_(b)
        phi, p, _ = s["ctx"].rk2_step(s["phi"], s["now"], s["dt"], solid=s["solid"], rho_air=RHO_AIR,
                                      rho_water=RHO_WATER, tol=TOL, forces=s["forces"])
        return {"u": s["now"], "phi": phi, "p": p}
    beta = mgproj.face_coeffs(s["phi"], s["h"], s["solid"], RHO_AIR, RHO_WATER, out=s["beta"])
    if s["grid"] == "stretched":
        beta, _ = mgproj.stretched_metrics(*s["widths"], beta)
    s["ctx"].update(beta)
    u, p, _ = s["ctx"].project(s["u"], dt=s["dt"], tol=TOL)
    return {"u": u, "p": p}


def work(case):
    """Each input read once, each output written once; the operations of one evaluation of the formulas around
    the solve and of one residual, which no solver can do without."""
    n = case["nx"] * case["ny"] * case["nz"]
    solid = n if case["body"] else 0
    if case["kind"] == "solve":
        return {"bytes": 8 * n * 5, "flops": 15 * n}                    # beta (3), rhs; p
    if case["kind"] == "momentum":
        return {"bytes": 8 * n * 10, "flops": 134 * n}                  # phi, beta, u; R
    if case["kind"] == "gradient":
        return {"bytes": 8 * n * 15 + solid, "flops": 100 * n}          # phi, u*, w; u, p, grad_u, grad_phi
    if case["kind"] == "step":
        return {"bytes": 8 * n * 9 + solid, "flops": 400 * n}           # phi, u; u, phi, p
    extra = {"uniform": 0, "cut": 24 * n, "stretched": 0}[case["grid"]]
    return {"bytes": 8 * n * 8 + extra + solid, "flops": 45 * n}        # phi, u*; u, p


# ---------------------------------------------------------------------------
# the same results in 64 bits, in plain torch
# ---------------------------------------------------------------------------
def _face_coeffs(phi, open_):
    rho = RHO_AIR + (RHO_WATER - RHO_AIR) * phi
    out = []
    for a, o in zip((2, 1, 0), open_):
        n = phi.shape[a] - 1
        b = torch.zeros_like(phi)
        b.narrow(a, 1, n).copy_(2.0 / (rho.narrow(a, 0, n) + rho.narrow(a, 1, n)))
        out.append(b * o)
    return tuple(out)


def _grad(p, h):
    out = []
    for a in (2, 1, 0):
        g = torch.zeros_like(p)
        n = p.shape[a] - 1
        torch.sub(p.narrow(a, 1, n), p.narrow(a, 0, n), out=g.narrow(a, 1, n))
        out.append(g.div_(h))
    return tuple(out)


def _div(f, h):
    d = torch.zeros_like(f[0])
    for a, x in zip((2, 1, 0), f):
        n = x.shape[a] - 1
        d.sub_(x)
        d.narrow(a, 0, n).add_(x.narrow(a, 1, n))
    return d.div_(h)


def _solve(coef, b, h):
    """The mean-free solution of D(coef G p) = b by conjugate gradients with the diagonal as preconditioner."""
    def diag():
        d = torch.zeros_like(b)
        for a, x in zip((2, 1, 0), coef):
            n = x.shape[a] - 1
            d.add_(x)
            d.narrow(a, 0, n).add_(x.narrow(a, 1, n))
        return d
    dg = diag()
    live = dg > 0
    inv = torch.where(live, h * h / torch.where(live, dg, torch.ones_like(dg)), torch.zeros_like(dg))
    cells = live.sum()
    mean_free = lambda v: torch.where(live, v - torch.where(live, v, torch.zeros_like(v)).sum() / cells, torch.zeros_like(v))
    r = -mean_free(b)  # of -A, which is positive semi-definite
    p = torch.zeros_like(b)
    stop = 1.0e-14 * float(torch.linalg.vector_norm(r))
    z = inv * r
    d, rz = z.clone(), torch.dot(r.flatten(), z.flatten())
    for it in range(20000):
        g = _grad(d, h)
        q = -_div(tuple(c * x for c, x in zip(coef, g)), h)
        alpha = rz / torch.dot(d.flatten(), q.flatten())
        p += alpha * d
        r -= alpha * q
        if it % 50 == 49 and float(torch.linalg.vector_norm(r)) <= stop:
            break
        torch.mul(inv, r, out=z)
        new = torch.dot(r.flatten(), z.flatten())
        d.mul_(new / rz).add_(z)
        rz = new
    return mean_free(p)


def _shift(v, axis, by):
    """v at the index moved by -1, 0 or 1 along axis, the outermost layer mirrored."""
    n = v.shape[axis]
    if by == 0:
        return v
    if by < 0:
        return torch.cat((v.narrow(axis, 0, 1), v.narrow(axis, 0, n - 1)), axis)
    return torch.cat((v.narrow(axis, 1, n - 1), v.narrow(axis, n - 1, 1)), axis)


def _up(v, axis):
    """The next value along axis, 0 beyond the last."""
    n = v.shape[axis]
    return torch.cat((v.narrow(axis, 1, n - 1), torch.zeros_like(v.narrow(axis, 0, 1))), axis)


def _down(v, axis):
    n = v.shape[axis]
    return torch.cat((torch.zeros_like(v.narrow(axis, 0, 1)), v.narrow(axis, 0, n - 1)), axis)


def _momentum(phi, beta, u, h):
    f = FORCES
    mu = f["mu_air"] + (f["mu_water"] - f["mu_air"]) * phi
    axes = (2, 1, 0)
    conv, visc = [], []
    for i, a in enumerate(axes):
        up = _up(u[i], a)
        c, t = (0.5 * (u[i] + up)) ** 2, 2.0 * mu * (up - u[i]) / h
        conv.append((c - _down(c, a)) / h)
        visc.append(t - _down(t, a))
    for i, a in enumerate(axes):
        for j, b in enumerate(axes):
            if j <= i:
                continue
            ui, uj = _shift(u[i], b, -1), _shift(u[j], a, -1)
            e = 0.25 * (mu + _shift(mu, a, -1) + _shift(mu, b, -1) + _shift(_shift(mu, a, -1), b, -1))
            flux = 0.25 * (u[j] + uj) * (u[i] + ui)
            shear = e * ((u[i] - ui) + (u[j] - uj)) / h
            conv[i] = conv[i] + (_up(flux, b) - flux) / h
            visc[i] = visc[i] + (_up(shear, b) - shear)
            conv[j] = conv[j] + (_up(flux, a) - flux) / h
            visc[j] = visc[j] + (_up(shear, a) - shear)
    out = []
    for i in range(3):
        r = -conv[i] + f["inv_re"] * beta[i] * visc[i] / h
        r = r - f["g"] if i == 2 else r
        out.append(torch.where(beta[i] > 0, r, torch.zeros_like(r)))
    return tuple(out)


def _vof(open_, u, phi, h, dt):
    flux = []
    for a, o, x in zip((2, 1, 0), open_, u):
        low = _shift(phi, a, -1)
        flux.append(o * x * torch.where(x > 0, low, phi))
    return dt * _div(tuple(flux), h)


def _projected(coef, beta, area, u, h, dt):
    """The velocity and the pressure of one projection; coef = area * beta."""
    p = _solve(coef, _div(tuple(a * x for a, x in zip(area, u)), h) / dt, h)
    g = _grad(p, h)
    return tuple(x - dt * b * y * (c > 0) for x, b, y, c in zip(u, beta, g, coef)), p


def exact(case, seed):
    n = case["nx"] * case["ny"] * case["nz"]
    if case["grid"] == "cut" or n > 2 ** 24 or (case["kind"] == "step" and n > 2 ** 21):
        return None  # the areas have no closed form here; the others would take too long
    d = _inputs(case, seed)
    phi, h, dt = d["phi"], d["h"], d["dt"]
    open_ = _open(phi.shape, d["solid"])
    beta = _face_coeffs(phi, open_)
    if case["kind"] == "solve":
        return {"p": _solve(beta, d["rhs"], h)}
    if case["kind"] == "momentum":
        return {"R": _momentum(phi, beta, d["u"], h)}
    if case["kind"] == "gradient":
        u, p = _projected(beta, beta, open_, d["u"], h, dt)
        q = _solve(beta, _div(tuple(b * x for b, x in zip(beta, d["w"])), h), h)
        gq = tuple(g * o for g, o in zip(_grad(q, h), open_))
        gu = tuple(w - g for w, g in zip(d["w"], gq))
        gphi = torch.zeros_like(phi)
        for a, b, g, t in zip((2, 1, 0), beta, _grad(p, h), gu):
            m = phi.shape[a] - 1
            x = b * b * (-dt * g * t)
            gphi.add_(x)
            gphi.narrow(a, 0, m).add_(x.narrow(a, 1, m))
        return {"u": u, "p": p, "grad_u": gu, "grad_phi": -0.5 * (RHO_WATER - RHO_AIR) * gphi}
    if case["kind"] == "step":
        ut = tuple(x + dt * r for x, r in zip(d["u"], _momentum(phi, beta, d["u"], h)))
        us, _ = _projected(beta, beta, open_, ut, h, dt)
        phis = phi - _vof(open_, d["u"], phi, h, dt)
        beta2 = _face_coeffs(phis, open_)
        ut = tuple(a + b + dt * r for a, b, r in zip(us, d["u"], _momentum(phis, beta2, us, h)))
        u1, p = _projected(beta2, beta2, open_, ut, h, dt)
        uh = tuple(0.5 * (a + b) for a, b in zip(us, d["u"]))
        return {"u": tuple(0.5 * x for x in u1), "phi": phi - _vof(open_, uh, phi, h, dt), "p": p}
    area = open_
    if case["grid"] == "stretched":
        w = [v.view(s) for v, s in zip(d["widths"], ((1, 1, -1), (1, -1, 1), (-1, 1, 1)))]
        area = tuple(o * a * b for o, a, b in zip(open_, (w[1], w[0], w[0]), (w[2], w[2], w[1])))
        mid = lambda v: 0.5 * (v + torch.cat((v[:1], v[:-1])))
        beta = tuple(b / mid(v).view(s) for b, v, s in zip(beta, d["widths"], ((1, 1, -1), (1, -1, 1), (-1, 1, 1))))
        h = 1.0
    u, p = _projected(tuple(a * b for a, b in zip(area, beta)), beta, area, d["u"], h, dt)
    return {"u": u, "p": p}
