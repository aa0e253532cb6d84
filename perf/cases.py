"""The calls a program makes of the library, as cases to time and compare: what each stands for is said beside it.

Every case builds a mesh and a permeability field from its own sizes (one reservoir), and its data from the seed (one
request on that reservoir): the hierarchy is kept from call to call, as a program that solves for several right-hand
sides keeps it. Cases of the "request" kind bring a mesh of their own each time. Iterative calls run either to a
tolerance that pins their result to rounding (1e-12 for a whole solve) or for a fixed number of inner iterations, so
that results can be compared.
"""
import math

import numpy as np
import torch

from paper_2005_01275_gb300 import nlmg

KIND = {"exp": nlmg.KAPPA_EXP, "inv": nlmg.KAPPA_INV1P2}


# ---- meshes and data ------------------------------------------------------------------------------------------

class Mesh:
    """A cell graph in the layout of the library: a box of unit cells' faces, Dirichlet on both ends of x."""

    def __init__(self, shape, perm, active=None, links=None):
        shape = tuple(shape)
        n = int(np.prod(shape))
        idx = np.arange(n).reshape(shape, order="F")
        h = np.array([1.0 / s for s in shape])
        keep = np.ones(n, bool) if active is None else active
        new = np.full(n, -1, np.int64)
        new[keep] = np.arange(int(keep.sum()))
        cells, half, tags, areas = [], [], [], []
        for ax in range(len(shape)):
            area = float(np.prod(np.delete(h, ax)))
            lo = np.take(idx, np.arange(shape[ax] - 1), axis=ax).reshape(-1)
            hi = np.take(idx, np.arange(1, shape[ax]), axis=ax).reshape(-1)
            both = keep[lo] & keep[hi]
            lo, hi = lo[both], hi[both]
            cells.append(np.stack([new[lo], new[hi]], 1))
            half.append(np.stack([perm[lo], perm[hi]], 1) * (2.0 * area / h[ax]))
            tags.append(np.zeros(lo.size))
            areas.append(np.full(lo.size, area))
        if links is not None:   # connections across a fault: pairs of cells that are no neighbours of the box
            lo, hi, mult = links
            both = keep[lo] & keep[hi]
            lo, hi, mult = lo[both], hi[both], mult[both]
            cells.append(np.sort(np.stack([new[lo], new[hi]], 1), axis=1))
            half.append(np.stack([perm[np.minimum(lo, hi)], perm[np.maximum(lo, hi)]], 1) * mult[:, None])
            tags.append(np.zeros(lo.size))
            areas.append(np.ones(lo.size))
        for ax in range(len(shape)):
            area = float(np.prod(np.delete(h, ax)))
            for side in (0, shape[ax] - 1):
                c = np.sort(np.take(idx, side, axis=ax).reshape(-1))
                c = c[keep[c]]
                cells.append(np.stack([new[c], np.full(c.size, -1)], 1))
                half.append(np.stack([perm[c] * (2.0 * area / h[ax]), np.zeros(c.size)], 1))
                tags.append(np.full(c.size, 1 if ax == 0 else 2))
                areas.append(np.full(c.size, area))
        self.n_cells = int(keep.sum())
        self.cell_volume = np.full(self.n_cells, float(np.prod(h)))
        self.face_cells = np.concatenate(cells).astype(np.int32)
        self.half_trans = np.ascontiguousarray(np.concatenate(half))
        self.face_bc = np.concatenate(tags).astype(np.uint8)
        self.face_area = np.concatenate(areas)
        self.n_faces = int(self.face_cells.shape[0])
        where = np.stack(np.unravel_index(np.nonzero(keep)[0], shape, order="F"), 1)
        self.x = (where + 0.5) * h


def _noise(shape, corr, rng):
    """A smooth random field of unit variance with a correlation length in cells."""
    k2 = sum(k * k for k in np.meshgrid(*[2 * np.pi * np.fft.fftfreq(s) for s in shape], indexing="ij"))
    v = np.real(np.fft.ifftn(np.fft.fftn(rng.standard_normal(shape)) * np.exp(-0.25 * k2 * corr ** 2)))
    return (v - v.mean()) / v.std()


def _perm(shape, decades, rng):
    """log-normal (decades = 0: sigma 1), or sinuous channels in a background over so many decades."""
    v = _noise(shape, 4.0, rng)
    if not decades:
        return np.exp(v).reshape(-1, order="F")
    ax = [np.arange(s) + 0.5 for s in shape]
    for _ in range(12):
        width, y0, phase = rng.uniform(2, 4), rng.uniform(0, shape[1]), rng.uniform(0, 2 * np.pi)
        yc = y0 + rng.uniform(0.1, 0.3) * shape[1] * np.sin(2 * np.pi * ax[0] / (rng.uniform(0.5, 1.5) * shape[0]) + phase)
        d2 = (ax[1][None, :, None] - yc[:, None, None]) ** 2 + (ax[2][None, None, :] - rng.uniform(0, shape[2])) ** 2
        v = v + 3.0 * np.exp(-2.0 * d2 / width ** 2)
    v = (v - v.min()) / (v.max() - v.min())
    return (10.0 ** (decades * (v - 0.5))).reshape(-1, order="F")


def _mesh(case, seed):
    rng = np.random.default_rng(seed)
    shape = tuple(case[k] for k in ("nx", "ny", "nz") if case.get(k))
    perm = _perm(shape, case.get("decades", 0), rng)
    if not case.get("faulted"):
        return Mesh(shape, perm)
    # one cell in sixteen is inactive, and a fault plane joins cells of neighbouring columns with a throw of two
    n = int(np.prod(shape))
    active = rng.uniform(size=n) > 1 / 16
    i = np.arange(n)
    x, z = i % shape[0], i // (shape[0] * shape[1])
    lo = i[(x == shape[0] // 2) & (z + 2 < shape[2])]
    hi = lo + 1 + 2 * shape[0] * shape[1]
    return Mesh(shape, perm, active, (lo, hi, rng.uniform(0.05, 0.5, lo.size)))


def _data(mesh, seed):
    """Dirichlet values on the two ends and a smooth source: one request."""
    rng = np.random.default_rng(seed)
    d = np.nonzero(mesh.face_bc == 1)[0]
    g = np.zeros(mesh.n_faces)
    g[d] = np.where(mesh.x[mesh.face_cells[d, 0], 0] < 0.5, rng.uniform(0.5, 1.5), rng.uniform(-0.5, 0.5))
    f = np.zeros(mesh.n_cells)
    for _ in range(4):
        c = rng.uniform(0.2, 0.8, mesh.x.shape[1])
        f += rng.uniform(-0.5, 0.5) * np.exp(-((mesh.x - c) ** 2).sum(1) / 0.02)
    return f, g


def _point(mesh, seed):
    """A pressure to linearise at: a smooth profile with some roughness."""
    rng = np.random.default_rng([seed, 1])
    return 1.0 - mesh.x[:, 0] + 0.2 * np.sin(2 * np.pi * mesh.x[:, -1]) * rng.uniform(0.5, 1.0) + 0.02 * rng.standard_normal(mesh.n_cells)


def _options(case):
    """Aggregates and modes as in this repository's workloads: 64 then 8 cells with 4 modes in 3D, 16 then 8 with 2 in 2D."""
    three = bool(case.get("nz"))
    o = dict(n_levels=3, agg_size=[64 if three else 16] + [8] * 6, modes=[4 if three else 2] * 7, dp_clamp=math.log(1.5) / case["a"] if case["kappa"] == "exp" else 0.5,
             smoother=case.get("smoother", "picard"), lin_precision=case.get("precision", 0), lin_precond=case.get("precond", 0))
    if case.get("faulted"):
        o["modes"] = [3] * 7
    if case.get("cap"):
        o["lin_maxit"] = case["cap"]
    return o


_kept = {}


def _reservoir(case):
    """The mesh and its hierarchy, kept from request to request."""
    key = tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "rows", "streams", "level")))
    if key not in _kept:
        mesh = _mesh(case, 7)
        _kept[key] = (mesh, nlmg.Context(mesh, KIND[case["kappa"]], case["a"], nlmg.options_from_dict(_options(case))))
    return _kept[key]


# ---- cases ----------------------------------------------------------------------------------------------------

def listed():
    return [
        # the residual on caller buffers that an application checks its own iterate with: the smallest mesh of the
        # repository, where a call is its launches, and a million cells
        dict(name="residual_32x32", kind="residual", nx=32, ny=32, kappa="exp", a=0.5),
        dict(name="residual_100x100x100", kind="residual", nx=100, ny=100, nz=100, kappa="exp", a=2.0, decades=6),
        # one multigrid cycle with a fixed number of inner iterations, as a smoother or inside another iteration
        dict(name="cycle_64x64x64", kind="cycle", nx=64, ny=64, nz=64, kappa="exp", a=2.0, decades=6, cap=25),
        # one coarse Picard step of that hierarchy on its own
        dict(name="coarse_64x64x64", kind="picard", level=1, nx=64, ny=64, nz=64, kappa="exp", a=2.0, decades=6, cap=40),
        # the frozen-coefficient linear system to full accuracy, multigrid-preconditioned, and the Newton system
        dict(name="linear_80x61x47", kind="picard", level=0, nx=80, ny=61, nz=47, kappa="exp", a=2.0, decades=6, precond=1),
        dict(name="newton_48x48x48", kind="newton", nx=48, ny=48, nz=48, kappa="exp", a=1.0, decades=4),
        # whole solves: the smallest configuration, the 64^3 workload in plain FP64, an unstructured mesh with FP32
        # inner solves, a million cells with the multigrid preconditioner
        dict(name="solve_32x32", kind="solve", nx=32, ny=32, kappa="exp", a=0.5),
        dict(name="solve_64x64x64", kind="solve", nx=64, ny=64, nz=64, kappa="exp", a=2.0, decades=6, smoother="picard_newton"),
        dict(name="solve_faulted", kind="solve", nx=45, ny=38, nz=27, kappa="inv", a=1.0, decades=3, faulted=True, precision=1),
        dict(name="solve_100x100x100", kind="solve", nx=100, ny=100, nz=100, kappa="exp", a=2.0, decades=6, smoother="picard_newton", precond=1, precision=2),
        # eight right-hand sides on eight streams, the batched mixed form the benchmark reports
        dict(name="many_64x64x64", kind="many", rows=8, streams=8, nx=64, ny=64, nz=64, kappa="exp", a=2.0, decades=6, smoother="picard_newton", precond=1, precision=2),
        # requests with meshes of their own through the request loop: the hierarchy is part of the call
        dict(name="request_65x63", kind="request", rows=4, nx=65, ny=63, kappa="exp", a=1.0),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["residual", "cycle", "coarse", "linear", "newton", "solve", "solve", "many", "request"])
    a = round(rng.uniform(0.5, 2.0), 3)
    if kind == "request" or (kind in ("residual", "solve") and rng.random() < 0.3):
        nx, ny = size(31, 90 if kind == "request" else 400), size(31, 90 if kind == "request" else 400)
        case = dict(kind=kind, nx=nx, ny=ny, kappa=rng.choice(["exp", "inv"]), a=a)
        return dict(case, rows=rng.randint(1, 4)) if kind == "request" else case
    cells = size(8000, 1000000 if kind in ("residual", "solve") else 300000)
    nx = int(round(cells ** (1 / 3) * rng.uniform(0.8, 1.25)))
    ny = int(round(cells ** (1 / 3) * rng.uniform(0.8, 1.25)))
    case = dict(kind=kind, nx=nx, ny=ny, nz=max(12, min(int(cells / (nx * ny)), 1000000 // (nx * ny))), kappa="exp", a=a, decades=rng.randint(3, 6))
    if kind == "cycle":
        case.update(cap=rng.randint(10, 30))
    elif kind == "coarse":
        case.update(kind="picard", level=rng.randint(1, 2), cap=rng.randint(10, 40))
    elif kind == "linear":
        case.update(kind="picard", level=0, precond=1)
    elif kind == "newton":
        case.update(a=round(rng.uniform(0.5, 1.0), 3), decades=rng.randint(2, 4))
    elif kind == "many":
        case.update(rows=rng.randint(2, 8), streams=rng.choice([2, 4, 8]), smoother="picard_newton", precond=1, precision=rng.choice([0, 2]))
    elif kind == "solve":
        if cells > 150000 or rng.random() < 0.4:
            case.update(smoother="picard_newton", precond=1, precision=rng.choice([0, 2]))
        else:
            case.update(smoother=rng.choice(["picard", "picard_newton"]), precision=rng.choice([0, 1]))
    return case


# ---- one pass -------------------------------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "request":
        meshes = [_mesh(case, 1000 * seed + r) for r in range(case["rows"])]
        reqs = [(m,) + _data(m, 1000 * seed + r) for r, m in enumerate(meshes)]
        return dict(case=case, reqs=reqs, opts=nlmg.options_from_dict(_options(case)),
                    server=nlmg.Server(max_inflight=4, setup_threads_per_request=2, hierarchy_cache=0))
    mesh, base = _reservoir(case)
    if kind in ("solve", "many"):
        rows = case.get("rows", 1)
        f, g = zip(*[_data(mesh, 1000 * seed + r) for r in range(rows)])
        s = dict(case=case, ctx=base, f=torch.from_numpy(np.stack(f)).cuda(), g=torch.from_numpy(np.stack(g)).cuda())
        s["p"] = torch.zeros_like(s["f"])
        return s
    f, g = _data(mesh, 1000 * seed)
    p = _point(mesh, seed)
    ctx = base.instance()
    ctx.set_data(f, g)
    s = dict(case=case, ctx=ctx, p=p)
    if kind == "residual":
        s.update(p=torch.from_numpy(p).cuda(), r=torch.zeros(mesh.n_cells, dtype=torch.float64, device="cuda"),
                 norm2=torch.zeros(1, dtype=torch.float64, device="cuda"))
    elif kind == "cycle":
        s["r0"] = float(np.linalg.norm(ctx.fine_residual(p)))
    elif kind == "picard" and case["level"] == 0:
        ctx.set_options(lin_tol=1e-13)
    elif kind == "picard":
        x = p
        for l in range(case["level"]):   # the point projected to the level, and a right-hand side near its operator's value
            x = ctx.transfer(l, nlmg.PROJECT, x)
        s["p"] = x
        s["b"] = ctx.level_apply(case["level"], x * (1.0 + 0.1 * np.sin(np.arange(x.size) + seed)))
        ctx.set_options(coarse_lin_tol=1e-6, coarsest_lin_tol=1e-6)
    elif kind == "newton":
        ctx.set_options(newton_lin_tol=1e-13)
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "residual":
        s["ctx"].fine_residual_noalloc(s["p"].data_ptr(), s["r"].data_ptr(), s["norm2"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        return s["r"], s["norm2"]
    if kind == "cycle":
        p, res, _ = s["ctx"].vcycle(s["p"], s["r0"])
        return p, res
    if kind == "picard":
        return s["ctx"].picard_update(case["level"], s["p"], s.get("b"))[0]
    if kind == "newton":
        return s["ctx"].newton_update(s["p"])[0]
    if kind == "solve":
        s["ctx"].solve_device(s["f"].data_ptr(), s["g"].data_ptr(), 0, s["p"].data_ptr(), tol_rel=1e-12, tol_abs=1e-300, max_cycles=60)
        return s["p"][0]
    if kind == "many":
        s["ctx"].solve_many_device(case["rows"], s["f"].data_ptr(), s["g"].data_ptr(), s["p"].data_ptr(), tol_rel=1e-12, tol_abs=1e-300, max_cycles=60, n_streams=case["streams"])
        return s["p"]
    tickets = [s["server"].submit(m, KIND[case["kappa"]], case["a"], s["opts"], f, g, tol_rel=1e-12, tol_abs=1e-300) for m, f, g in s["reqs"]]
    return [s["server"].poll(t, wait_ms=60000)[0] for t in tickets]


def work(case):
    """The mesh's arrays (per cell its volume, data and pressure; per face its cells, halves and data) read once and the
    result written; operations of one residual per row. A coarse level has about a sixteenth of the fine one's unknowns."""
    n = case["nx"] * case["ny"] * case.get("nz", 1)
    faces = (3 if case.get("nz") else 2) * n
    rows = case.get("rows", 1)
    if case["kind"] == "picard" and case["level"]:
        n, faces = n / 16 ** case["level"], faces / 16 ** case["level"]
    once = 8 * n + 24 * faces
    return {"bytes": once * (rows if case["kind"] == "request" else 1) + rows * 24 * n, "flops": rows * (20 * faces + 20 * n)}


# ---- the same in 64 bits, with torch alone --------------------------------------------------------------------

class _Plain:
    def __init__(self, mesh, kappa, a, f, g):
        t = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()  # noqa: E731
        fc, bc = mesh.face_cells.astype(np.int64), mesh.face_bc
        i, d, n = bc == 0, bc == 1, bc == 2
        self.K, self.L, self.u0, self.u1 = t(fc[i, 0]), t(fc[i, 1]), t(mesh.half_trans[i, 0]), t(mesh.half_trans[i, 1])
        self.D, self.ud, self.gd = t(fc[d, 0]), t(mesh.half_trans[d, 0]), t(g[d])
        self.rhs = t(mesh.cell_volume * f)
        self.rhs.index_add_(0, t(fc[n, 0]), t(mesh.face_area[n] * g[n]))
        self.kappa, self.a = kappa, a

    def kap(self, p):
        return torch.exp(self.a * p) if self.kappa == "exp" else 1.0 / (1.0 + p * p)

    def dkap(self, p):
        return self.a * torch.exp(self.a * p) if self.kappa == "exp" else -2.0 * p / (1.0 + p * p) ** 2

    def to_cells(self, on_faces, on_ends, sign=-1.0):
        return torch.zeros_like(self.rhs).index_add_(0, self.K, on_faces).index_add_(0, self.L, sign * on_faces).index_add_(0, self.D, on_ends)

    def freeze(self, p):
        k = self.kap(p)
        ha, hb = k[self.K] * self.u0, k[self.L] * self.u1
        return ha * (hb / (ha + hb)), k[self.D] * self.ud, ha, hb

    def residual(self, p):
        T, Td, _, _ = self.freeze(p)
        return self.to_cells(T * (p[self.K] - p[self.L]), Td * (p[self.D] - self.gd)) - self.rhs

    def picard(self, p):
        """The frozen matrix at p as a product, and its diagonal."""
        T, Td, _, _ = self.freeze(p)
        return (lambda v: self.to_cells(T * (v[self.K] - v[self.L]), Td * v[self.D])), self.to_cells(T, Td, 1.0)

    def newton(self, p):
        """The Jacobian of the residual at p as a product, and the frozen matrix's diagonal."""
        T, Td, ha, hb = self.freeze(p)
        dk, diff = self.dkap(p), p[self.K] - p[self.L]
        cK = T + (hb / (ha + hb)) ** 2 * dk[self.K] * self.u0 * diff
        cL = -T + (ha / (ha + hb)) ** 2 * dk[self.L] * self.u1 * diff
        cD = Td + dk[self.D] * self.ud * (p[self.D] - self.gd)
        return (lambda v: self.to_cells(cK * v[self.K] + cL * v[self.L], cD * v[self.D])), self.to_cells(T, Td, 1.0)


def _krylov(A, diag, b, tol, most=20000):
    """BiCGStab preconditioned by the diagonal, on new residuals until they fall no further; None where it does not get there."""
    x, best = torch.zeros_like(b), math.inf
    w = diag.rsqrt()
    goal = tol * float((w * b).norm())
    for _ in range(6):
        r = b - A(x)
        now = float((w * r).norm())
        if now <= goal or now > 0.5 * best:
            break
        best, rh, p, rho, it = now, r / diag, r.clone(), None, 0
        rho = rh @ r
        while it < most:
            v = A(p / diag)
            alpha = rho / (rh @ v)
            s = r - alpha * v
            t = A(s / diag)
            omega = (t @ (s / diag)) / (t @ (t / diag))
            x = x + alpha * (p / diag) + omega * (s / diag)
            r = s - omega * t
            new = rh @ r
            p = r + (new / rho) * (alpha / omega) * (p - omega * v)
            rho = new
            it += 1
            if it % 25 == 0 and not float((w * r).norm()) > 0.3 * goal:
                break
    return x if float((w * (b - A(x))).norm()) <= max(100 * goal, 1e-11 * float((w * b).norm())) else None


def _plain_solve(P, clamp):
    """Picard steps, then Newton steps, from zero to the rounding of the residual; None where they do not get there."""
    p = torch.zeros_like(P.rhs)
    r = P.residual(p)
    first = float(r.norm())
    for k in range(60):
        A, d = (P.picard if float(r.norm()) > 1e-2 * first else P.newton)(p)
        dx = _krylov(A, d, -r, 1e-6, 3000)
        if dx is None:
            return None
        p = p + dx * min(1.0, clamp / max(float(dx.abs().max()), 1e-300))
        r = P.residual(p)
        if float(r.norm()) <= 3e-14 * first:
            return p
        if k > 40 and float(r.norm()) <= 1e-12 * first:
            return p
    return None


def exact(case, seed):
    kind = case["kind"]
    n = case["nx"] * case["ny"] * case.get("nz", 1)
    if kind == "cycle" or (kind == "picard" and case["level"]) or (kind in ("solve", "many") and n * case.get("rows", 1) > 300000):
        return None
    if kind == "request":
        meshes = [_mesh(case, 1000 * seed + r) for r in range(case["rows"])]
    else:
        meshes = [_mesh(case, 7)] * case.get("rows", 1)
    data = [_data(m, 1000 * seed + r) for r, m in enumerate(meshes)]
    P = [_Plain(m, case["kappa"], case["a"], f, g) for m, (f, g) in zip(meshes, data)]
    if kind in ("solve", "many", "request"):
        clamp = _options(case)["dp_clamp"]
        out = [_plain_solve(q, clamp) for q in P]
        return out[0] if kind == "solve" else out if kind == "request" else None if any(o is None for o in out) else torch.stack(out)
    p = torch.from_numpy(_point(meshes[0], seed)).cuda()
    r = P[0].residual(p)
    if kind == "residual":
        return r, (r @ r).reshape(1)
    A, d = (P[0].newton if kind == "newton" else P[0].picard)(p)
    return _krylov(A, d, -r, 1e-13)
