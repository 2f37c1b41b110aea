"""Performance cases of the library's public calls, and what they should return.

Each case is one call (or one time step's calls) that a flow solver makes: pressure solves from
the smallest grids to 1024^3, a moving body's whole time step, batches, the velocity solves,
classification, the residual check and the surface forces.  ``listed()`` gives the named cases,
``draw()`` more of the same ranges; ``exact()`` recomputes a case's result in 64 bits with plain
torch from the method's definition (closed bodies; a dense eigenbasis of the empty box
preconditions GMRES).  Boxes have edges in proportion to their cell counts, so cells are near
isotropic where the grid is uniform and within the stretching elsewhere.
"""
import math

import numpy as np
import torch

import paper_2605_04335_gb300 as pkg

TOL = 1e-10


# ----------------------------------------------------------------------------- cases

def listed():
    return [
        # the smallest solve of the configurations: latency of a V-cycle's many short kernels
        {"name": "solve_sphere_64", "kind": "solve", "nx": 64, "ny": 64, "nz": 64, "ratio": 1.0, "body": "sphere",
         "precision": 1},
        # FP64 throughout (the paper's precision), odd and uneven extents
        {"name": "solve_fp64_193x161x129", "kind": "solve", "nx": 193, "ny": 161, "nz": 129, "ratio": 2.0,
         "body": "ellipsoid", "precision": 0},
        # the ordinary production size: stretched 256^3 with the double-FP32 refinement
        {"name": "solve_ellipsoid_256", "kind": "solve", "nx": 256, "ny": 256, "nz": 256, "ratio": 2.0,
         "body": "ellipsoid", "precision": 2},
        # the largest single-GPU grid, twelve bodies, FP64 refinement, the autotuner's schedule for it
        {"name": "solve_spheres_1024", "kind": "solve", "nx": 1024, "ny": 1024, "nz": 1024, "ratio": 1.0,
         "body": "spheres", "precision": 1, "omega": 1.2, "inner": 3},
        # a moving body's time step on the paper's subdomain shape: reclassify, datum, solve, forces
        {"name": "step_ellipsoid_301x385x129", "kind": "step", "nx": 301, "ny": 385, "nz": 129, "ratio": 2.0,
         "body": "ellipsoid", "precision": 2},
        # a flapping zero-thickness plate's time step: cut links, Krylov acceleration
        {"name": "step_plate_512", "kind": "step", "nx": 512, "ny": 512, "nz": 512, "ratio": 2.0, "body": "plate",
         "precision": 2},
        # the advection-diffusion solves of one time step: three velocity components, no-slip body
        {"name": "velocity_256", "kind": "velocity", "nx": 256, "ny": 256, "nz": 256, "ratio": 2.0,
         "body": "ellipsoid", "precision": 2},
        # many independent uneven problems advanced together
        {"name": "batch_48_edges_64_192", "kind": "batch", "count": 48, "lo": 64, "hi": 192, "draw": 5, "precision": 1},
        # many small problems: launches and their latency
        {"name": "batch_96_edges_16_32", "kind": "batch", "count": 96, "lo": 16, "hi": 32, "draw": 7, "precision": 2},
        # iblanking alone: new positions of twelve bodies, the tables read by the flow solver
        {"name": "classify_spheres_512", "kind": "classify", "nx": 512, "ny": 512, "nz": 512, "ratio": 1.0,
         "body": "spheres", "precision": 1},
        # the residual check of a field inside a time-step loop that may not allocate
        {"name": "residual_256", "kind": "residual", "nx": 256, "ny": 256, "nz": 256, "ratio": 2.0,
         "body": "ellipsoid", "precision": 0},
        # pressure forces on the structure's nodes: the smallest call of a step
        {"name": "forces_ellipsoid_256", "kind": "forces", "nx": 256, "ny": 256, "nz": 256, "ratio": 2.0,
         "body": "ellipsoid", "precision": 0},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def grid(lo, hi):
        n = log_int(lo, hi)
        return {a: max(lo // 2, min(hi, int(round(n * rng.uniform(0.6, 1.25))))) for a in ("nx", "ny", "nz")}

    kind = rng.choice(["solve", "solve", "solve", "step", "step", "velocity", "velocity", "batch", "batch", "classify",
                       "residual", "forces"])
    if kind == "batch":
        lo = log_int(16, 64)
        return {"kind": kind, "count": log_int(4, 48), "lo": lo, "hi": lo + log_int(8, 2 * lo), "draw": rng.randrange(1000),
                "precision": rng.choice([1, 2])}
    case = {"kind": kind, "ratio": rng.choice([1.0, 2.0]), "precision": rng.choice([1, 1, 2, 2, 0])}
    if kind == "step" and rng.random() < 0.4:
        case.update(grid(64, 320), body="plate", precision=rng.choice([1, 2]))
    elif kind in ("solve", "step", "velocity"):
        case.update(grid(32, 224 if case["precision"] == 0 else 448), body=rng.choice(["sphere", "ellipsoid"]))
    else:
        case.update(grid(48, 512), body=rng.choice(["sphere", "ellipsoid"]))
    return case


# ----------------------------------------------------------------------------- inputs

def _faces(n, ratio, length):
    """n + 1 faces on [0, length]; ratio: widest over narrowest cell (tanh map, finest at the centre)."""
    s = np.arange(n + 1) / n
    if ratio > 1.0:
        beta = math.acosh(math.sqrt(ratio))
        s[1:-1] = 0.5 + np.arctanh(np.tanh(beta) * (2.0 * s[1:-1] - 1.0)) / (2.0 * beta)
    return length * s


class _Mesh:
    def __init__(self, verts, tris, closed):
        self.verts, self.tris, self.closed = verts, tris, closed


def _ellipsoid(centre, semi, angle, nlat=33, nlon=128):
    """Latitude-longitude ellipsoid of 2 nlon (nlat - 1) triangles, turned by angle about z."""
    th = math.pi * np.arange(1, nlat) / nlat
    ph = 2.0 * math.pi * np.arange(nlon) / nlon
    ring = np.stack(np.broadcast_arrays(np.sin(th)[:, None] * np.cos(ph), np.sin(th)[:, None] * np.sin(ph),
                                        np.cos(th)[:, None]), -1).reshape(-1, 3)
    v = np.concatenate([[[0.0, 0.0, 1.0]], ring, [[0.0, 0.0, -1.0]]]) * np.asarray(semi)
    c, s = math.cos(angle), math.sin(angle)
    v = v @ np.array([[c, s, 0.0], [-s, c, 0.0], [0.0, 0.0, 1.0]]) + np.asarray(centre)
    a, b = np.arange(nlon), (np.arange(nlon) + 1) % nlon
    t = [np.stack([np.zeros(nlon, int), 1 + a, 1 + b], 1)]
    for r in range(nlat - 2):
        p, q = 1 + r * nlon, 1 + (r + 1) * nlon
        t += [np.stack([p + a, q + a, q + b], 1), np.stack([p + a, q + b, p + b], 1)]
    last, end = 1 + (nlat - 2) * nlon, 1 + (nlat - 1) * nlon
    t.append(np.stack([last + a, np.full(nlon, end), last + b], 1))
    return _Mesh(v, np.concatenate(t).astype(np.int32), 1)


def _plate(centre, chord, span, angle, nq=100):
    """Zero-thickness rectangle of 2 nq^2 triangles, pitched by angle about y."""
    g = np.arange(nq + 1) / nq - 0.5
    x, y = np.meshgrid(g * chord, g * span, indexing="xy")
    c, s = math.cos(angle), math.sin(angle)
    v = np.stack([c * x.ravel(), y.ravel(), -s * x.ravel()], 1) + np.asarray(centre)
    i = np.arange((nq + 1) ** 2).reshape(nq + 1, nq + 1)
    a, b, d, e = i[:-1, :-1].ravel(), i[:-1, 1:].ravel(), i[1:, 1:].ravel(), i[1:, :-1].ravel()
    return _Mesh(v, np.concatenate([np.stack([a, b, d], 1), np.stack([a, d, e], 1)]).astype(np.int32), 0)


def _geometry(case, seed, fixed=False):
    """Faces of the three axes and the body's meshes; the seed moves and turns the body a little."""
    n = (case["nx"], case["ny"], case["nz"])
    ext = [m / max(n) for m in n]
    faces = [_faces(m, case["ratio"], e) for m, e in zip(n, ext)]
    r = np.random.RandomState(seed % (1 << 31))
    mid = np.array([0.5 * e for e in ext])
    size = min(ext)
    if not fixed:
        mid = mid + 0.02 * size * (r.rand(3) - 0.5)
    turn = math.radians(20.0 + (0.0 if fixed else 5.0 * r.rand()))
    body = case["body"]
    if body == "sphere":
        meshes = [_ellipsoid(mid, (0.15 * size,) * 3, turn, 17, 64)]
    elif body == "ellipsoid":
        meshes = [_ellipsoid(mid, (0.3 * size, 0.13 * size, 0.13 * size), turn)]
    elif body == "plate":
        meshes = [_plate(mid, 0.4 * size, 0.2 * size, math.radians(30.0) * math.cos(turn))]
    else:   # twelve non-overlapping spheres on a jittered 3 x 2 x 2 lattice of the box
        meshes = []
        for q in range(12):
            cell = np.array([(q % 3 + 0.5) / 3.0, (q // 3 % 2 + 0.5) / 2.0, (q // 6 + 0.5) / 2.0]) * ext
            meshes.append(_ellipsoid(cell + 0.06 * size * (r.rand(3) - 0.5), (size * (0.03 + 0.05 * r.rand()),) * 3,
                                     0.0, 17, 64))
    return faces, meshes


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _divergence(faces, seed):
    """Discrete divergence of a random N(0, 1) velocity field (face value: mean of its two cells)."""
    g = _gen(seed)
    shape = tuple(len(f) - 1 for f in faces[::-1])
    b = torch.zeros(shape, dtype=torch.float64, device="cuda")
    for ax, f in enumerate(faces):
        d = 2 - ax
        h = torch.from_numpy(np.diff(f)).cuda().reshape([-1 if q == d else 1 for q in range(3)])
        u = torch.randn(shape, dtype=torch.float64, device="cuda", generator=g)
        n = shape[d]
        flux = 0.5 * (u.narrow(d, 0, n - 1) + u.narrow(d, 1, n - 1))
        del u
        b.narrow(d, 0, n - 1).add_(flux / h.narrow(d, 0, n - 1))
        b.narrow(d, 1, n - 1).sub_(flux / h.narrow(d, 1, n - 1))
        del flux
    return b


def _smooth(faces, seed, modes=3):
    """A smooth field: the product over the axes of 1 + a few cosines."""
    r = np.random.RandomState(seed % (1 << 31))
    out = None
    for f in faces[::-1]:
        x = torch.from_numpy(0.5 * (f[:-1] + f[1:])).cuda()
        v = torch.ones_like(x)
        for a, k, ph in r.rand(modes, 3):
            v = v + 0.5 * a / modes * torch.cos((1.0 + 6.0 * k) * x + 2.0 * math.pi * ph)
        out = v if out is None else out[..., None] * v
    return out.contiguous()


def _accel(meshes, seed):
    """Rigid accelerations: a0, angular acceleration, angular velocity, centre (per mesh)."""
    r = np.random.RandomState((seed + 3) % (1 << 31))
    return np.stack([np.concatenate([r.randn(3), 2.0 * r.randn(3), r.randn(3), m.verts.mean(0)]) for m in meshes])


def _velocity(meshes, seed):
    r = np.random.RandomState((seed + 4) % (1 << 31))
    return np.stack([np.concatenate([0.3 * r.randn(3), r.randn(3), m.verts.mean(0)]) for m in meshes])


def _alpha(faces):
    """Half a viscous time step: dt = half the smallest width at unit speed, Reynolds number 1000."""
    return 0.5 * min(float(np.diff(f).min()) for f in faces) / 2000.0


def _batch_cases(case):
    r = np.random.RandomState(case["draw"])
    out = []
    for _ in range(case["count"]):
        n = r.randint(case["lo"], case["hi"] + 1, 3)
        out.append({"nx": int(n[0]), "ny": int(n[1]), "nz": int(n[2]), "ratio": 1.0,
                    "body": "sphere" if r.rand() < 0.5 else "ellipsoid"})
    return out


# ----------------------------------------------------------------------------- state and pass

_ctx = None


class _State:
    """One program's handles and buffers; the tables are given back with it."""

    def __init__(self, case):
        global _ctx
        if _ctx is None:
            _ctx = pkg.Context(0)
        self.case, self.ctx, self.tables = case, _ctx, []
        self.opts = pkg.SolveOpts(precision=case["precision"], omega=case.get("omega", 1.3),
                                  inner_cycles=case.get("inner", 2))

    def classify(self, faces, meshes):
        t = pkg.Tables(self.ctx, *faces, meshes)
        self.tables.append(t)
        return t

    def __del__(self):
        for t in self.tables:
            t.close()


def prepare(case, seed):
    s = _State(case)
    kind, prec = case["kind"], case["precision"]
    if kind == "batch":
        s.rhs, cells = [], 0
        for q, c in enumerate(_batch_cases(case)):
            faces, meshes = _geometry(c, seed + q)
            t = s.classify(faces, meshes)
            pkg.ibm_smoother_sweeps(s.ctx.h, t.h, prec, 1)      # the solver's arrays for these tables
            s.rhs.append(_divergence(faces, seed + 101 * q))
            cells += t.ncell
        s.all = torch.zeros(cells, dtype=torch.float64, device="cuda")
        s.p = [v.reshape(b.shape) for v, b in zip(s.all.split([b.numel() for b in s.rhs]), s.rhs)]
        return s
    s.faces, s.meshes = _geometry(case, seed)
    if kind in ("step", "classify"):   # the tables of the body's position one step ago
        s.t = s.classify(s.faces, _geometry(case, seed, fixed=True)[1])
    else:
        s.t = s.classify(s.faces, s.meshes)
    if kind in ("solve", "step"):
        pkg.ibm_smoother_sweeps(s.ctx.h, s.t.h, prec, 1)
        s.rhs = _divergence(s.faces, seed)
        s.p = torch.zeros_like(s.rhs)
        s.motion = _accel(s.meshes, seed)
    elif kind == "velocity":
        s.alpha = _alpha(s.faces)
        s.u0 = torch.stack([_smooth(s.faces, seed + 11 * c) for c in range(3)])
        s.u = s.u0.clone()
        s.f = s.u0 + 0.1 * torch.stack([_smooth(s.faces, seed + 11 * c + 5) for c in range(3)])
        s.motion = _velocity(s.meshes, seed)
        pkg.ibm_helmholtz_sweeps_timed(s.ctx.h, s.t.h, s.alpha, prec, 1, s.f[0], s.u[0])
    elif kind == "classify":   # a flow solver's own table arrays, with room for every body position
        room = case["nx"] * case["ny"] + case["ny"] * case["nz"] + case["nx"] * case["nz"]
        f64, i64, i32 = torch.float64, torch.int64, torch.int32
        s.out = {k: torch.zeros(shape, dtype=t, device="cuda") for k, shape, t in (
            ("iblank", s.t.shape, torch.uint8), ("cell", room, i64), ("bi", (room, 3), f64), ("ip", (room, 3), f64),
            ("base", (room, 3), i32), ("flags", room, i32), ("ref", (room, 8), i64), ("w", (room, 8), f64),
            ("scale", room, f64))}
    elif kind in ("residual", "forces"):
        s.rhs = _divergence(s.faces, seed)
        s.p = _smooth(s.faces, seed + 7)
        s.motion = _accel(s.meshes, seed)
        s.export = s.t.export()    # the residual check reads the tables from the caller's arrays
    return s


def run(s):
    kind = s.case["kind"]
    if kind == "solve":
        s.p.zero_()
        s.t.solve(s.rhs, s.p, TOL, s.opts)
        return {"p": s.p}
    if kind == "step":
        s.t.reclassify(s.meshes)
        s.t.neumann_rigid(s.motion)
        s.p.zero_()
        s.t.solve(s.rhs, s.p, TOL, s.opts)
        return {"p": s.p, **s.t.surface_forces(s.meshes, s.p, motions=s.motion)}
    if kind == "velocity":
        s.u.copy_(s.u0)
        ub = s.t.boundary_velocity_rigid(s.motion)
        for c in range(3):
            s.t.helmholtz_solve(s.alpha, s.f[c], s.u[c], ub[c].contiguous(), TOL,
                                pkg.HelmholtzOpts(precision=s.case["precision"]))
        return {"u": s.u}
    if kind == "batch":
        s.all.zero_()
        pkg.poisson_solve_batched(s.ctx.h, [t.h for t in s.tables], s.rhs, TOL, s.p, s.opts)
        return {"p": s.all}
    if kind == "classify":
        s.t.reclassify(s.meshes)
        pkg.ibm_tables_export(s.t.h, **s.out)
        return s.out
    if kind == "residual":
        e = s.export
        return list(torch.tensor(pkg.ibm_residual_norm_noalloc(*s.faces, e["iblank"], e["cell"], e["ref"], e["w"],
                                                               e["scale"], s.rhs, s.p), dtype=torch.float64))
    return s.t.surface_forces(s.meshes, s.p, motions=s.motion)


def work(case):
    """Bytes: the call's arrays, each read or written once (a grid of FP64 values and its mask).
    Operations: one residual per row (14), what a solve needs to know that it is done."""
    if case["kind"] == "batch":
        cells = sum(c["nx"] * c["ny"] * c["nz"] for c in _batch_cases(case))
    else:
        cells = case["nx"] * case["ny"] * case["nz"]
    tris = {"sphere": 2048, "ellipsoid": 8192, "plate": 20000, "spheres": 12 * 2048}.get(case.get("body"), 0)
    per_cell = {"solve": 17, "batch": 17, "step": 18, "velocity": 73, "classify": 1, "residual": 17, "forces": 0}
    flops = {"solve": 14, "batch": 14, "step": 14, "velocity": 45, "classify": 0, "residual": 14, "forces": 0}
    return {"bytes": per_cell[case["kind"]] * cells + 200 * tris, "flops": flops[case["kind"]] * cells + 200 * tris}


# ----------------------------------------------------------------------------- 64-bit results

class _Box:
    """The 7-point operator of a stretched box with closed walls, and its eigenbasis."""

    def __init__(self, faces):
        self.faces = [torch.from_numpy(f).cuda() for f in faces]
        self.c = [0.5 * (f[1:] + f[:-1]) for f in self.faces]
        self.h = [f[1:] - f[:-1] for f in self.faces]
        self.cm, self.cp, self.basis, lam = [], [], [], []
        for c, h in zip(self.c, self.h):
            gap = c[1:] - c[:-1]
            cm, cp = torch.zeros_like(h), torch.zeros_like(h)
            cm[1:], cp[:-1] = 1.0 / (h[1:] * gap), 1.0 / (h[:-1] * gap)
            self.cm.append(cm)
            self.cp.append(cp)
            w = h.sqrt()
            off = 1.0 / (gap * (h[1:] * h[:-1]).sqrt())
            ev, q = torch.linalg.eigh(torch.diag(-(cm + cp)) + torch.diag(off, 1) + torch.diag(off, -1))
            ev[-1] = 0.0                                   # the constant
            lam.append(ev)
            self.basis.append((q.T * w, q / w[:, None]))
        self.lam = lam[2][:, None, None] + lam[1][None, :, None] + lam[0]
        self.vol = self.h[2][:, None, None] * self.h[1][None, :, None] * self.h[0]

    @staticmethod
    def _along(x, m, d):
        return torch.movedim(torch.movedim(x, d, -1) @ m.T, -1, d)

    def invert(self, x, inv):
        for d in range(3):
            x = self._along(x, self.basis[2 - d][0], d)
        x = x * inv
        for d in range(3):
            x = self._along(x, self.basis[2 - d][1], d)
        return x.contiguous()

    def apply(self, x):
        y = torch.zeros_like(x)
        for d in range(3):
            n, shape = x.shape[d], [-1 if q == d else 1 for q in range(3)]
            diff = x.narrow(d, 1, n - 1) - x.narrow(d, 0, n - 1)
            y.narrow(d, 0, n - 1).add_(diff * self.cp[2 - d][:-1].reshape(shape))
            y.narrow(d, 1, n - 1).sub_(diff * self.cm[2 - d][1:].reshape(shape))
        return y


def _base(c, v):
    i = (torch.searchsorted(c, v.contiguous(), right=True) - 1).clamp(0, c.numel() - 2)
    return i, ((v - c[i]) / (c[i + 1] - c[i])).clamp(0.0, 1.0)


def _corners(box, x, shape):
    """Linear cells (n, 8) and trilinear weights of points x (n, 3)."""
    (i, tx), (j, ty), (k, tz) = (_base(box.c[a], x[:, a]) for a in range(3))
    cell, w = [], []
    for q in range(8):
        a, b, d = q & 1, q >> 1 & 1, q >> 2
        cell.append(((k + d) * shape[1] + j + b) * shape[2] + i + a)
        w.append((tx if a else 1 - tx) * (ty if b else 1 - ty) * (tz if d else 1 - tz))
    return torch.stack(cell, 1), torch.stack(w, 1)


def _closest(p, tri):
    """Closest points of a surface (triangles (m, 3, 3)) to points p (n, 3)."""
    out = torch.empty_like(p)
    a, ab, ac = tri[:, 0], tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0]
    g11, g12, g22 = (ab * ab).sum(1), (ab * ac).sum(1), (ac * ac).sum(1)
    det = g11 * g22 - g12 * g12
    for s in range(0, len(p), 1024):
        x = p[s:s + 1024, None]
        ap = x - a
        d, e = (ap * ab).sum(2), (ap * ac).sum(2)
        u, v = (g22 * d - g12 * e) / det, (g11 * e - g12 * d) / det
        best = a + u[..., None] * ab + v[..., None] * ac
        dist = ((x - best) ** 2).sum(2).masked_fill(~((u >= 0) & (v >= 0) & (u + v <= 1)), math.inf)
        for q in range(3):
            p0, edge = tri[:, q], tri[:, (q + 1) % 3] - tri[:, q]
            t = (((x - p0) * edge).sum(2) / (edge * edge).sum(1)).clamp(0.0, 1.0)
            y = p0 + t[..., None] * edge
            dy = ((x - y) ** 2).sum(2)
            near = dy < dist
            best, dist = torch.where(near[..., None], y, best), torch.where(near, dy, dist)
        m = dist.argmin(1)
        out[s:s + 1024] = best[torch.arange(len(m), device=p.device), m]
    return out


class _Rows:
    """Convex closed bodies on a box: fluid cells, ghost cells and their image-point rows."""

    def __init__(self, box, meshes):
        self.box = box
        cx, cy, cz = box.c
        self.shape = shape = (len(cz), len(cy), len(cx))
        dev = cx.device

        def snapped(v):   # the inside test works on a lattice of 2^-24
            return torch.round(v * 2.0 ** 24)
        solid = torch.zeros(shape, dtype=torch.bool, device=dev)
        tris = []
        for m in meshes:
            v = torch.from_numpy(np.ascontiguousarray(m.verts)).to(dev)
            tri = v[torch.from_numpy(m.tris.astype(np.int64)).to(dev)]
            tris.append(tri)
            t = snapped(tri)
            n = torch.linalg.cross(t[:, 1] - t[:, 0], t[:, 2] - t[:, 0])
            rng = [torch.nonzero((c >= v[:, a].min()) & (c <= v[:, a].max())).flatten() for a, c in enumerate(box.c)]
            if min(len(r) for r in rng) == 0:
                continue
            k, j, i = torch.meshgrid(rng[2], rng[1], rng[0], indexing="ij")
            pts = snapped(torch.stack([cx[i], cy[j], cz[k]], -1).reshape(-1, 3))
            inside = torch.cat([((q @ n.T) < (t[:, 0] * n).sum(1)).all(1) for q in pts.split(8192)])
            solid[k.flatten(), j.flatten(), i.flatten()] |= inside
        self.tri = torch.cat(tris)
        self.fluid = ~solid
        near = torch.zeros_like(solid)
        for d in range(3):
            n = shape[d]
            near.narrow(d, 0, n - 1).logical_or_(self.fluid.narrow(d, 1, n - 1))
            near.narrow(d, 1, n - 1).logical_or_(self.fluid.narrow(d, 0, n - 1))
        ghost = solid & near
        g = torch.nonzero(ghost.flatten()).flatten()
        self.cell = g
        known = (self.fluid | ghost).flatten()
        self.active = self.fluid | ghost
        i, j, k = g % shape[2], g // shape[2] % shape[1], g // (shape[1] * shape[2])
        gc = torch.stack([cx[i], cy[j], cz[k]], 1)
        self.bi = _closest(gc, self.tri)
        ip = 2 * self.bi - gc
        ref, w = _corners(box, ip, shape)
        w = torch.where(known[ref], w, 0.0)
        total = w.sum(1, keepdim=True)
        w = w / total
        own = (ref == g[:, None])
        ws = torch.where(own, w, 0.0).sum(1)
        back = (total[:, 0] < 1e-3) | (ws >= 1 - 1e-12)       # rows that copy a fluid neighbour
        ws = torch.where(back, 0.0, ws)
        w = torch.where(own, 0.0, w) / (1 - ws)[:, None]
        best, far = torch.zeros_like(g), torch.full_like(ws, math.inf)
        scale = torch.zeros_like(ws)
        flat = self.fluid.flatten()
        for ax, step in ((0, 1), (1, shape[2]), (2, shape[1] * shape[2])):
            idx, n = (i, j, k)[ax], shape[2 - ax]
            for sgn in (-1, 1):
                ok = (idx + sgn >= 0) & (idx + sgn < n)
                nb = torch.where(ok, g + sgn * step, g)
                ok &= flat[nb]
                pos = gc.clone()
                pos[:, ax] = box.c[ax][(idx + sgn).clamp(0, n - 1)]
                d2 = ((ip - pos) ** 2).sum(1)
                take = ok & (d2 < far)
                best, far = torch.where(take, nb, best), torch.where(take, d2, far)
                coef = (box.cp if sgn < 0 else box.cm)[ax][(idx + sgn).clamp(0, n - 1)]
                scale += torch.where(ok, coef, 0.0)
        first = torch.zeros_like(ref, dtype=torch.bool)
        first[:, 0] = True
        self.ref = torch.where(back[:, None], best[:, None], ref)
        self.w = torch.where(back[:, None], first.to(w.dtype), w)
        self.ws, self.scale = ws, scale
        to = torch.stack([cx[best % shape[2]], cy[best // shape[2] % shape[1]], cz[best // (shape[1] * shape[2])]], 1)
        self.dir = torch.where(back[:, None], to - gc, ip - gc)
        self.length = self.dir.norm(dim=1)
        self.dir = self.dir / self.length[:, None]

    def interp(self, x):
        return (self.w * x.flatten()[self.ref]).sum(1)

    def mean(self, x):
        v = torch.where(self.fluid, self.box.vol, 0.0)
        return (v * x).sum() / v.sum()

    def gauge(self, x):
        return torch.where(self.active, x - self.mean(x), 0.0)


def _gmres(op, pre, b, n=90, restarts=4):
    """Right-preconditioned GMRES to the floor of FP64 (vectors are flat tensors)."""
    x = torch.zeros_like(b)
    for _ in range(restarts):
        r = b - op(x)
        beta = r.norm()
        if float(beta) <= 2e-14 * float(b.norm()):
            break
        q, z, hess = [r / beta], [], np.zeros((n + 1, n))
        for k in range(n):
            z.append(pre(q[k]))
            w = op(z[k])
            for _ in range(2):
                for a in range(k + 1):
                    d = torch.dot(q[a], w)
                    w.sub_(d * q[a])
                    hess[a, k] += float(d)
            hess[k + 1, k] = float(w.norm())
            q.append(w / hess[k + 1, k])
            rhs = np.zeros(k + 2)
            rhs[0] = float(beta)
            y, *_ = np.linalg.lstsq(hess[:k + 2, :k + 1], rhs, rcond=None)
            left = np.linalg.norm(hess[:k + 2, :k + 1] @ y - rhs)
            if left < 1e-8 * float(beta) or left < 1e-14 * float(b.norm()):
                break
        for v, c in zip(z, y):
            x.add_(v, alpha=float(c))
    return x


def _pressure(rows, rhs, datum=None):
    """The zero-mean pressure: fluid rows A p + lambda = rhs, ghost rows g - sum w v = datum."""
    box, fl = rows.box, rows.fluid
    inv = torch.where(box.lam.abs() < 1e-9 * box.lam.abs().max(), 0.0, 1.0 / box.lam)
    inv[~torch.isfinite(inv)] = 0.0
    row_scale = rows.scale

    def op(v):
        x, lam = v[:-1].reshape(rows.shape), v[-1]
        y = torch.where(fl, box.apply(x) + lam, x).flatten()
        y[rows.cell] = row_scale * (x.flatten()[rows.cell] - rows.interp(x))
        return torch.cat([y, rows.mean(x)[None]])

    def pre(v):
        r = v[:-1].reshape(rows.shape)
        z = box.invert(torch.where(fl, r, 0.0), inv)
        y = torch.where(rows.active, z, r).flatten()
        y[rows.cell] += v[:-1][rows.cell] / row_scale
        return torch.cat([y, v[-1:]])

    b = torch.where(fl, rhs, 0.0).flatten()
    b = b - rows.fluid.flatten() * rows.mean(rhs)
    if datum is not None:
        b[rows.cell] = row_scale * datum
    x = _gmres(op, pre, torch.cat([b, b.new_zeros(1)]))
    return rows.gauge(x[:-1].reshape(rows.shape))


def _velocity_field(rows, alpha, f, ub):
    """(I - alpha A) u = f with the boundary value at the midpoint of each ghost and its image."""
    box, fl = rows.box, rows.fluid
    inv = 1.0 / (1.0 - alpha * box.lam)

    def op(v):
        x = v.reshape(rows.shape)
        y = torch.where(fl, x - alpha * box.apply(x), x).flatten()
        y[rows.cell] = (1 + rows.ws) * v[rows.cell] + (1 - rows.ws) * rows.interp(x)
        return y

    def pre(v):
        r = v.reshape(rows.shape)
        z = torch.where(fl, box.invert(torch.where(fl, r, 0.0), inv), r).flatten()
        z[rows.cell] = (v[rows.cell] - (1 - rows.ws) * rows.interp(z)) / (1 + rows.ws)
        return z

    b = torch.where(fl, f, 0.0).flatten()
    b[rows.cell] = 2.0 * ub
    return _gmres(op, pre, b).reshape(rows.shape)


def _rigid(points, motion):
    """Acceleration of a rigid body's points: a0 + alpha x r + omega x (omega x r)."""
    m = torch.from_numpy(motion).to(points.device)
    r = points - m[9:12]
    al, om = m[3:6].expand_as(r), m[6:9].expand_as(r)
    return m[:3] + torch.linalg.cross(al, r) + torch.linalg.cross(om, torch.linalg.cross(om, r))


def _forces(rows, meshes, p, motion):
    """Pressure at 1.5 cell diagonals off each triangle, less its normal gradient, and the
    nodes' thirds of each triangle's force (one closed body)."""
    tri = rows.tri
    area = torch.linalg.cross(tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0])
    n = area / area.norm(dim=1, keepdim=True)
    c = tri.mean(1)
    cell = [(torch.searchsorted(f, c[:, a].contiguous(), right=True) - 1).clamp(0, len(f) - 2)
            for a, f in enumerate(rows.box.faces)]
    d = 1.5 * torch.stack([rows.box.h[a][cell[a]] for a in range(3)], 1).norm(dim=1)
    ref, w = _corners(rows.box, c + d[:, None] * n, rows.shape)
    w = torch.where(rows.fluid.flatten()[ref], w, 0.0)
    total = w.sum(1)
    q = -(_rigid(c, motion[0]) * n).sum(1)
    ps = torch.where(total >= 1e-3, (w * p.flatten()[ref]).sum(1) / total - d * q, 0.0)
    share = -(ps[:, None] * area) / 6.0
    node = torch.zeros((len(meshes[0].verts), 3), dtype=p.dtype, device=p.device)
    idx = torch.from_numpy(meshes[0].tris.astype(np.int64)).to(p.device)
    for a in range(3):
        node.index_add_(0, idx[:, a], share)
    return {"p_side": torch.stack([ps, torch.zeros_like(ps)], 1), "flags": None, "f_node": node}


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        cs = _batch_cases(case)
        if sum(c["nx"] * c["ny"] * c["nz"] for c in cs) > 2 ** 23 or case["count"] > 48:
            return None                                    # many dense eigenbases: over 20 seconds
        out = []
        for q, c in enumerate(cs):
            faces, meshes = _geometry(c, seed + q)
            out.append(_pressure(_Rows(_Box(faces), meshes), _divergence(faces, seed + 101 * q)).flatten())
        return {"p": torch.cat(out)}
    # cut links and exact tables have no short 64-bit statement; GMRES on larger grids takes over 20 seconds
    if case["body"] in ("plate", "spheres") or kind == "classify" or case["nx"] * case["ny"] * case["nz"] > 2 ** 24:
        return None
    faces, meshes = _geometry(case, seed)
    rows = _Rows(_Box(faces), meshes)
    if kind == "velocity":
        m = torch.from_numpy(_velocity(meshes, seed)[0]).cuda()
        r = rows.bi - m[6:9]
        ub = (m[:3] + torch.linalg.cross(m[3:6].expand_as(r), r)).T.contiguous()
        u = []
        for c in range(3):
            f = _smooth(faces, seed + 11 * c) + 0.1 * _smooth(faces, seed + 11 * c + 5)
            u.append(_velocity_field(rows, _alpha(faces), f, ub[c]))
        return {"u": torch.stack(u)}
    rhs = _divergence(faces, seed)
    motion = _accel(meshes, seed)
    if kind == "residual":
        p = _smooth(faces, seed + 7)
        r = torch.where(rows.fluid, rhs - rows.box.apply(p), 0.0)
        ghost = rows.scale * (rows.interp(p) - p.flatten()[rows.cell])
        a = torch.where(rows.fluid, r - rows.mean(r), 0.0).square().sum() + ghost.square().sum()
        b = torch.where(rows.fluid, rhs - rows.mean(rhs), 0.0).square().sum()
        return [(a / b).sqrt(), a.sqrt(), b.sqrt()]
    if kind == "forces":
        return _forces(rows, meshes, _smooth(faces, seed + 7), motion)
    if kind == "solve":
        return {"p": _pressure(rows, rhs)}
    datum = (rows.dir * _rigid(rows.bi, motion[0])).sum(1) * rows.length / (1 - rows.ws)
    p = _pressure(rows, rhs, datum)
    return {"p": p, **_forces(rows, meshes, p, motion)}
