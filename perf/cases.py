"""The work a user of the pressure multigrid has it do, as cases with sizes.

A case is one call (or one small group of calls) through the public entry
points of ``paper_1410_8568_gb300.gbmg``, on seeded two-phase fields: a liquid
film with a drop above it (periodic in x and y, walls in z) or spheres in a
closed box, density ratios from 10 to 1000, smooth velocity divergences or
white noise on the right.  Kinds:

``step``        one time step of a flow solver: the new density goes to the
                handle (faces, coarse faces, coarsest grid), then a cold-start
                solve to 1e-10;
``projection``  one projection step: the non-projected velocity in, S = D u/dt,
                the solve from the last pressure, the velocity corrected;
``host``        the same time step for a program whose arrays are host memory;
``batch``       many small grids of uneven sizes solved together;
``serve``       requests of uneven sizes handed to the serving loop and awaited.
"""
import math

import numpy as np
import torch

from paper_1410_8568_gb300 import gbmg

TOL = 1e-10
NEUMANN, PERIODIC = gbmg.NEUMANN, gbmg.PERIODIC


def case(name, kind="step", nx=0, ny=0, nz=0, field="drop", ratio=1000.0, precision="mixed",
         solver="mg", prolongation="trilinear", outer="fp64", count=1, lo=0, hi=0):
    c = {"name": name, "kind": kind, "nx": nx, "ny": ny, "nz": nz, "field": field, "ratio": ratio,
         "precision": precision, "solver": solver, "prolongation": prolongation, "outer": outer,
         "count": count, "lo": lo, "hi": hi}
    if name is None:
        del c["name"]
    return c


def listed():
    return [
        # the smallest production grid: a sphere in a closed box; launches and latency
        case("step_32", nx=32, ny=32, nz=32, field="sphere"),
        # the drop/film field at an everyday size, and the two sizes above it
        case("step_128", nx=128, ny=128, nz=128),
        case("step_256", nx=256, ny=256, nz=256),
        case("step_512", nx=512, ny=512, nz=512),
        # every level in FP64
        case("fp64_128", nx=128, ny=128, nz=128, precision="fp64"),
        # a box that is not a cube, flux-conserving prolongation
        case("flux_192x128x96", nx=192, ny=128, nz=96, prolongation="flux", ratio=100.0),
        # conjugate gradients with the V-cycle as preconditioner
        case("pcg_96", nx=96, ny=96, nz=96, solver="pcg"),
        # an edge with a large odd factor: the hierarchy stops at 25^3
        case("odd_100", nx=100, ny=100, nz=100, field="sphere", ratio=100.0),
        # Chorin's projection around the solve, from the last step's pressure
        case("projection_192", kind="projection", nx=192, ny=192, nz=192),
        # density and right-hand side arrive in pinned host memory
        case("host_128", kind="host", nx=128, ny=128, nz=128),
        # independent spheres of uneven sizes in one launch
        case("batch_24", kind="batch", count=24, lo=32, hi=128, field="sphere"),
        # uneven requests in flight together in the serving loop
        case("serve_8", kind="serve", count=8, lo=64, hi=256),
    ]


def _smooth_edge(rng, lo, hi):
    """An edge m 2^k, m in {2, 3} (an exact coarsest grid), about log-uniform."""
    edges = sorted(m << k for m in (2, 3) for k in range(0, 10) if lo <= (m << k) <= hi)
    u = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(edges, key=lambda e: abs(math.log(e / u)))


def _odd_edges(rng):
    """Three edges with odd factors up to 25 (a larger coarsest grid)."""
    k = rng.choice((1, 2, 2, 3))
    top = 25 if k < 3 else 21
    return [rng.choice(range(5, top + 1, 2)) << k for _ in range(3)]


def draw(rng):
    kind = rng.choice(("step",) * 10 + ("projection", "host", "batch", "serve"))
    ratio = round(math.exp(rng.uniform(math.log(10.0), math.log(1000.0))), 3)
    field = rng.choice(("drop", "sphere"))
    if kind == "batch":
        hi = rng.choice((64, 96, 128))
        return case(None, kind=kind, count=rng.randint(3, 32), lo=rng.choice((16, 32)), hi=hi, field="sphere",
                    ratio=ratio)
    if kind == "serve":
        return case(None, kind=kind, count=rng.randint(2, 10), lo=rng.choice((32, 48, 64)),
                    hi=rng.choice((128, 192, 256)), ratio=ratio)
    if kind in ("projection", "host"):
        n = _smooth_edge(rng, 32, 256)
        return case(None, kind=kind, nx=n, ny=_smooth_edge(rng, n / 2, n), nz=_smooth_edge(rng, n / 2, n), field=field,
                    ratio=ratio)
    mode = rng.choice(("mixed",) * 5 + ("odd",) * 2 + ("xp", "fp64", "pcg", "flux"))
    if mode == "odd":
        nx, ny, nz = _odd_edges(rng)
        return case(None, nx=nx, ny=ny, nz=nz, field=field, ratio=ratio)
    n = _smooth_edge(rng, 16, 384 if mode in ("mixed", "xp") else 192)
    nx, ny, nz = n, _smooth_edge(rng, max(8, n / 2), n), _smooth_edge(rng, max(8, n / 2), n)
    return case(None, nx=nx, ny=ny, nz=nz, field=field, ratio=ratio,
                precision="fp64" if mode == "fp64" else "mixed", solver="pcg" if mode == "pcg" else "mg",
                prolongation="flux" if mode == "flux" else "trilinear", outer="xp" if mode == "xp" else "fp64")


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _bc(field):
    return (PERIODIC, PERIODIC, NEUMANN) if field == "drop" else (NEUMANN, NEUMANN, NEUMANN)


def _edges(c, rng):
    """Grid sizes of a batch or a stream: cubes, log-uniform between lo and hi.
    The largest size is always there; the others come from the case alone."""
    sizes = [e for e in (16, 24, 32, 48, 64, 96, 128, 192, 256) if c["lo"] <= e <= c["hi"]]
    out = [sizes[-1]]
    for _ in range(c["count"] - 1):
        u = math.exp(rng.uniform(math.log(sizes[0]), math.log(sizes[-1])))
        out.append(min(sizes, key=lambda e: abs(math.log(e / u))))
    return [(n, n, n) for n in out]


def _shapes(c):
    if c["kind"] in ("batch", "serve"):
        return _edges(c, np.random.default_rng(1000 * c["count"] + c["hi"]))
    return [(c["nx"], c["ny"], c["nz"])]


def _centres(n):
    return (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) / n


def _length(shape):
    """Domain lengths: cubic cells, the longest edge 1."""
    return tuple(n / max(shape) for n in shape)


def _density(shape, field, ratio, rng):
    """Drop over a film, or a sphere in a box (in fractions of the edges); tanh interface over about 3 cells."""
    nx, ny, nz = shape
    x, y, z = _centres(nx)[None, None, :], _centres(ny)[None, :, None], _centres(nz)[:, None, None]
    eps = 1.5 / max(shape)
    drops = []
    if field == "drop":
        drops.append(((0.5 + rng.uniform(-0.05, 0.05), 0.5 + rng.uniform(-0.05, 0.05), rng.uniform(0.28, 0.36)), 0.125))
        for _ in range(int(rng.integers(0, 4))):
            drops.append(((rng.uniform(0.1, 0.9), rng.uniform(0.1, 0.9), rng.uniform(0.6, 0.9)), rng.uniform(0.02, 0.05)))
        d = (z - 0.1).expand(nz, ny, nx)
    else:
        drops.append((tuple(rng.uniform(0.3, 0.7, 3)), rng.uniform(0.1, 0.2)))
        d = torch.full((1, 1, 1), float("inf"), dtype=torch.float64, device="cuda").expand(nz, ny, nx)
    for (cx, cy, cz), r in drops:
        d = torch.minimum(d, ((x - cx) ** 2 + (y - cy) ** 2 + (z - cz) ** 2).sqrt_().sub_(r))
    return d.div(-eps).tanh_().add_(1.0).mul_(0.5 * (ratio - 1.0)).add_(1.0).contiguous()


def _velocity(shape, bc, rng):
    """Random smooth MAC velocity (8 Fourier modes), low-face layout, no flow through walls."""
    n = shape
    k = rng.integers(1, 5, size=(8, 3))
    amp = rng.standard_normal((8, 3))
    phase = rng.uniform(0.0, 2.0 * math.pi, size=8)
    out = []
    for comp in range(3):
        e = []
        for ax in range(3):
            q = torch.arange(n[ax], dtype=torch.float64, device="cuda")
            q = (q if ax == comp else q + 0.5) / n[ax]
            a = 2.0 * math.pi * torch.from_numpy(k[:, ax].astype(np.float64)).cuda()[:, None] * q[None, :]
            e.append((torch.cos(a), torch.sin(a)))
        (cx, sx), (cy, sy), (cz, sz) = e
        w = torch.from_numpy(amp[:, comp]).cuda()
        ph = torch.from_numpy(phase).cuda()
        # sin(kx + ky + kz + phi) = Im of the product: two rank-8 matrix products over (z, (y x))
        pc, ps = torch.cos(ph) * w, torch.sin(ph) * w
        cxy = (cy[:, :, None] * cx[:, None, :] - sy[:, :, None] * sx[:, None, :]).reshape(8, -1)
        sxy = (sy[:, :, None] * cx[:, None, :] + cy[:, :, None] * sx[:, None, :]).reshape(8, -1)
        zc = pc[:, None] * cz - ps[:, None] * sz
        zs = pc[:, None] * sz + ps[:, None] * cz
        u = (zs.T @ cxy + zc.T @ sxy).reshape(n[2], n[1], n[0])
        if bc[comp] == NEUMANN:
            u.select(2 - comp, 0).zero_()
        out.append(u.contiguous())
    return out


def _divergence(u, bc, shape, dt):
    """(high face - low face) / h summed over the axes, over dt; the high wall carries no flow."""
    s = torch.zeros_like(u[0])
    for d in range(3):
        ax = 2 - d
        s += (torch.roll(u[d], -1, ax) - u[d]) * max(shape)  # a wall's stored low face is 0: the roll brings that 0 to the high wall
    return s / dt


def _problem(shape, field, ratio, seed):
    rng = np.random.default_rng(seed)
    rho = _density(shape, field, ratio, rng)
    bc = _bc(field)
    if field == "drop":
        rhs = _divergence(_velocity(shape, bc, rng), bc, shape, 1.0)
    else:
        g = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 40)))
        rhs = torch.randn(rho.shape, dtype=torch.float64, device="cuda", generator=g)
    return bc, rho, rhs - rhs.mean()


def _solver(c, shape, bc, rho):
    return gbmg.Solver(shape, bc, rho=rho, length=_length(shape),
                       precision=gbmg.FP64 if c["precision"] == "fp64" else gbmg.MIXED,
                       solver=gbmg.SOLVER_PCG if c["solver"] == "pcg" else gbmg.SOLVER_MG,
                       prolongation=gbmg.PROLONG_FLUX if c["prolongation"] == "flux" else gbmg.PROLONG_TRILINEAR,
                       outer=gbmg.OUTER_XP if c["outer"] == "xp" else gbmg.OUTER_FP64)


DT = 1e-3


def _inputs(c, seed):
    return [_problem(s, c["field"], c["ratio"], [seed, g]) for g, s in enumerate(_shapes(c))]


def prepare(c, seed):
    kind, shapes = c["kind"], _shapes(c)
    made = _inputs(c, seed)
    st = {"kind": kind}
    if kind == "serve":
        st["server"] = gbmg.Server(32 << 30, max_slots=8)
        st["asks"] = []
        for shape, (bc, rho, rhs) in zip(shapes, made):
            faces = [torch.empty_like(rho) for _ in range(3)]
            gbmg.faces_from_density(shape, bc, rho, *faces)  # cubes of edge 1, as the requests are
            st["asks"].append((shape, bc, faces, rhs, torch.zeros_like(rhs)))
        return st
    # the handles exist since the last time step: they hold its density
    before = [_density(s, c["field"], c["ratio"], np.random.default_rng([seed, g, 1])) for g, s in enumerate(shapes)]
    st["solvers"] = [_solver(c, s, bc, old) for s, (bc, _, _), old in zip(shapes, made, before)]
    st["rho"] = [m[1] for m in made]
    st["rhs"] = [m[2] for m in made]
    if kind == "host":
        st["host"] = [torch.empty(t.shape, dtype=torch.float64, pin_memory=True) for t in (st["rho"][0], st["rhs"][0], st["rhs"][0])]
        st["host"][0].copy_(st["rho"][0])
        st["host"][1].copy_(st["rhs"][0])
        return st
    st["p"] = [torch.zeros_like(b) for b in st["rhs"]]
    if kind == "batch":
        st["batch"] = gbmg.Batch(st["solvers"])
    if kind == "projection":
        st["ustar"], st["p0"] = _flow(c, seed)
        st["u"] = [torch.empty_like(a) for a in st["ustar"]]
        st["S"] = torch.empty_like(st["p0"])
    return st


def _flow(c, seed):
    shape, bc = (c["nx"], c["ny"], c["nz"]), _bc(c["field"])
    rng = np.random.default_rng([seed, 2])
    return _velocity(shape, bc, rng), 100.0 * _velocity(shape, (PERIODIC,) * 3, rng)[0]


def run(st):
    kind = st["kind"]
    if kind == "serve":
        for _, _, _, _, p in st["asks"]:
            p.zero_()
        torch.cuda.current_stream().synchronize()  # the server's streams are its own
        tickets = [st["server"].submit(shape, bc, faces, rhs, p, tol=TOL) for shape, bc, faces, rhs, p in st["asks"]]
        st["server"].drain()
        for t in tickets:
            st["server"].poll(t)
        return [a[4] for a in st["asks"]]
    if kind == "host":
        rho, rhs, p = (t.numpy() for t in st["host"])
        p.fill(0.0)
        st["solvers"][0].step_host(rho, rhs, p, tol=TOL)
        return [p]
    for s, rho in zip(st["solvers"], st["rho"]):
        s.set_density(rho)
    if kind == "projection":
        p = st["p"][0]
        p.copy_(st["p0"])
        for a, b in zip(st["u"], st["ustar"]):
            a.copy_(b)
        st["solvers"][0].projection_step(st["u"], DT, p, st["S"], tol=TOL)
        return {"p": p, "u": st["u"], "S": st["S"]}
    for p in st["p"]:
        p.zero_()
    if kind == "batch":
        st["batch"].solve(st["rhs"], st["p"], tol=TOL)
    else:
        st["solvers"][0].solve(st["rhs"][0], st["p"][0], tol=TOL)
    return st["p"]


def work(c):
    """The inputs in and the solution out, and one application of the operator
    (13 operations a cell); what a solve does beyond that is its method."""
    cells = sum(x * y * z for x, y, z in _shapes(c))
    per = {"serve": 40, "projection": 80}.get(c["kind"], 24)  # serve: three face arrays in; projection: three velocities in and out
    return {"bytes": per * cells, "flops": 13 * cells}


# ---------------------------------------------------------------------------
# the same answers in 64 bits, by conjugate gradients in plain torch
# ---------------------------------------------------------------------------

def _faces(rho, bc, shape):
    """2 / (rho_low + rho_high) / h^2 per axis on low faces, 0 at walls."""
    w = []
    for d in range(3):
        ax = 2 - d
        f = (2.0 * max(shape) ** 2) / (rho + torch.roll(rho, 1, ax))
        if bc[d] == NEUMANN:
            f.select(ax, 0).zero_()
        w.append(f)
    return w


def _exact_solve(shape, bc, rho, rhs, most=40000):
    w = _faces(rho, bc, shape)

    def minus_a(x):
        y = torch.zeros_like(x)
        for d in range(3):
            ax = 2 - d
            f = w[d] * (x - torch.roll(x, 1, ax))
            y += f - torch.roll(f, -1, ax)
        return y

    diag = sum(f + torch.roll(f, -1, 2 - d) for d, f in enumerate(w))
    b = rhs.mean() - rhs
    x = torch.zeros_like(b)
    r = b.clone()
    bn = float(b.norm())
    z = r / diag
    p = z.clone()
    rz = (r * z).sum()
    for it in range(1, most + 1):
        q = minus_a(p)
        a = rz / (p * q).sum()
        x += a * p
        r -= a * q
        if it % 50 == 0:
            if it % 500 == 0:
                r = b - minus_a(x)
                r -= r.mean()
            if float(r.norm()) <= 1e-13 * bn:
                break
        z = r / diag
        new = (r * z).sum()
        p = z + (new / rz) * p
        rz = new
    return x - x.mean()


def exact(c, seed):
    shapes = _shapes(c)
    if sum(x * y * z for x, y, z in shapes) > 2.5e7:
        return None  # conjugate gradients would take over 20 seconds
    made = _inputs(c, seed)
    if c["kind"] == "projection":
        shape, (bc, rho, _) = shapes[0], made[0]
        ustar, _ = _flow(c, seed)
        S = _divergence(ustar, bc, shape, DT)
        p = _exact_solve(shape, bc, rho, S)
        u = [a - DT * (w / max(shape)) * (p - torch.roll(p, 1, 2 - d))
             for d, (a, w) in enumerate(zip(ustar, _faces(rho, bc, shape)))]
        return {"p": p, "u": u, "S": S}
    out = [_exact_solve(s, bc, rho, rhs) for s, (bc, rho, rhs) in zip(shapes, made)]
    return [p.cpu().numpy() for p in out] if c["kind"] == "host" else out
