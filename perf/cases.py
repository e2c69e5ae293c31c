"""The work that users of this library have it do, as measurable cases.

Each case goes through the public Python binding.  Geometries, operators, contexts and the network are what a program
keeps; level sets, right-hand sides and fields are inputs, made on the GPU from the seed.  Grids are those of the
repository's workloads (spheres and ellipsoids of 16^3 to 192^3, the 9-cell cavity up to 96 x 96 x 1152, batches of
32^3 to 64^3 cavities) and grids of unequal sides, cut to a cavity's bounding box as a careful user would."""
import math

import torch

import paper_1301_3794_gb300 as dm

CELL, EQUATOR, IRIS = 0.1154, 0.1033, 0.035   # the 9-cell cavity of the repository's workloads, metres


def listed():
    return [
        # one operator product on a small grid, in a loop that may not allocate: launch latency counts
        _case("apply_sphere32", "apply_noalloc", "sphere", 32, 32, 32),
        # the FP64 operator on its own, as a residual check or a user's own Krylov loop calls it
        _case("apply_ellipsoid128", "apply", "ellipsoid", 128, 128, 128),
        # checking a set of eigenpairs from elsewhere (another run, a file) against the operator
        _case("certify_ragged", "certify", "ellipsoid", 88, 72, 104, nev=8),
        # removing the divergent part of a field, a grid of unequal sides
        _case("project_ragged_f32", "project", "ellipsoid", 104, 88, 72, precision="f32"),
        # one shifted solve with everything in FP64, a middle-sized grid of unequal sides
        _case("solve_ragged_f64", "solve", "ellipsoid", 72, 56, 88, precision="f64", sigma=3.0),
        # one shifted solve with the BF16 V-cycle
        _case("solve_sphere128_bf16", "solve", "sphere", 128, 128, 128, precision="bf16", sigma=5.0),
        # one shifted solve of the benchmark's cavity: the inner step of its eigensolve
        _case("solve_ellipsoid192_f32", "solve", "ellipsoid", 192, 192, 192, precision="f32", sigma=5.0),
        # one shifted solve of the long accelerating structure, the largest grid of the repository
        _case("solve_ninecell_f32", "solve", "ninecell", 96, 96, 1152, precision="f32", sigma=0.0),
        # one step of training the learned smoother on the structure's residuals (forward, backward, Adam)
        _case("train_ninecell48", "train", "ninecell", 48, 48, 576, precision="f32", sigma=0.0),
        # the smallest whole job: level set to four modes in FP64
        _case("modes_sphere16_f64", "modes", "sphere", 16, 16, 16, precision="f64", sigma=7.0, nev=4),
        # an ordinary whole job: level set to eight modes with the FP32 V-cycle
        _case("modes_ellipsoid96_f32", "modes", "ellipsoid", 96, 96, 96, precision="f32", sigma=5.0, nev=8),
        # a sweep over small cavities of uneven size on worker streams
        _case("batch_32_64_f32", "batch", "mixed", 64, 64, 64, precision="f32", nev=5, count=6),
    ]


def _case(name, call, shape, nx, ny, nz, precision="f64", sigma=5.0, nev=1, count=1):
    c = {"call": call, "shape": shape, "nx": nx, "ny": ny, "nz": nz, "precision": precision, "sigma": sigma,
         "nev": nev, "count": count}
    return {"name": name, **c} if name else c


def draw(rng):
    call = rng.choice(["apply_noalloc", "apply", "certify", "project", "project", "solve", "solve", "solve", "train",
                       "modes", "modes", "batch"])

    def side(lo, hi):   # multiples of 8 (the multigrid halves a grid while it is even), even over the logarithm
        return 8 * round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 8)

    precision = rng.choice(["f64", "f32", "f32", "bf16"])
    sigma = round(rng.uniform(2.0, 6.0), 3)
    if call == "train" or (call == "solve" and rng.random() < 0.25):
        nxy = rng.choice([16, 32, 48] if call == "train" else [32, 48, 64, 80])
        # the structure's own proportions, and others: the spacing along z need not be that across
        nz = 16 * round(nxy * 12 * rng.uniform(0.6, 1.0) / 16)
        return _case("", call, "ninecell", nxy, nxy, nz, rng.choice(["f64", "f32", "f32"]) if call == "solve" else "f32", 0.0)
    if call == "batch":
        return _case("", call, "mixed", 64, 64, 64, "f32", 5.0, rng.randint(4, 7),
                     rng.randint(2, 6))
    if call == "modes":
        precision = rng.choice(["f64", "f32"])
        n = side(16, 48 if precision == "f64" else 88)
        return _case("", call, rng.choice(["sphere", "ellipsoid"]), n, n, n, precision, sigma, rng.randint(2, 8))
    hi = {"apply_noalloc": 88, "apply": 160, "certify": 128, "project": 144, "solve": 144}[call]
    nx = side(16, hi)
    ny, nz = (max(16, 8 * round(nx * rng.uniform(0.65, 1.0) / 8)) for _ in range(2))
    nev = rng.randint(1, 12) if call == "certify" else 1
    return _case("", call, rng.choice(["sphere", "ellipsoid"]) if nx == ny == nz else "ellipsoid", nx, ny, nz,
                 precision, sigma, nev)


def _gen(seed):
    return torch.Generator().manual_seed(int(seed) & 0x7FFFFFFF)


def _spacing(case):
    if case["shape"] == "ninecell":
        return (2.13 * EQUATOR / case["nx"], 2.13 * EQUATOR / case["ny"], 13.0 * CELL / case["nz"])
    return (2.2 / max(case["nx"], case["ny"], case["nz"]),) * 3


def _sigma(case):
    # below the lowest mode of the long structure, of the order of its smallest eigenvalue
    return case["sigma"] or 0.25 * (math.pi / (13.0 * CELL)) ** 2


def _nodes(case):
    h, n = _spacing(case), (case["nx"], case["ny"], case["nz"])
    z0 = -2.0 * CELL if case["shape"] == "ninecell" else -0.5 * n[2] * h[2]
    lo = (-0.5 * n[0] * h[0], -0.5 * n[1] * h[1], z0)
    x, y, z = (lo[a] + h[a] * torch.arange(n[a] + 1, dtype=torch.float64, device="cuda") for a in range(3))
    return x[None, None, :], y[None, :, None], z[:, None, None]


def _phi(case, g):
    """Level set at the nodes [nz+1][ny+1][nx+1], negative inside the cavity, from the generator g."""
    x, y, z = _nodes(case)
    if case["shape"] == "ninecell":
        # beam pipes of two cell lengths, nine cells whose equators vary by a percent; a smooth profile
        eq = EQUATOR * (1.0 + 0.01 * torch.randn(9, generator=g, dtype=torch.float64)).to("cuda")
        u = z / CELL
        r = IRIS + (eq[u.long().clamp(0, 8)] - IRIS) * torch.sin(math.pi * (u - u.floor())) ** 2
        r = torch.where((u > 0) & (u < 9), r, torch.full_like(r, IRIS))
        return torch.sqrt(x * x + y * y) - r
    h, n = _spacing(case), (case["nx"], case["ny"], case["nz"])
    off = torch.rand(3, generator=g, dtype=torch.float64).tolist()   # a sub-cell shift of the centre
    scale = 1.0
    if case["shape"] == "ellipsoid":
        scale = 0.6 + 0.4 * torch.rand(3, generator=g, dtype=torch.float64)
        scale = (scale / scale.max() if n[0] == n[1] == n[2] else 0.85 + 0.375 * (scale - 0.6)).tolist()
    semi = [n[a] * h[a] / 2.2 * (scale[a] if scale != 1.0 else 1.0) for a in range(3)]
    q = sum(((c - off[a] * h[a]) / semi[a]) ** 2 for a, c in enumerate((x, y, z)))
    return (torch.sqrt(q) - 1.0) * min(semi)


def _shapes(case):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    return (nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx)


def _field(case, g, count=1):
    """Face fields [count][F] of a few long waves and a little noise: what a Krylov basis or a stored mode holds."""
    h, out = _spacing(case), []
    n = (case["nx"], case["ny"], case["nz"])
    for _ in range(count):
        parts = []
        for s in _shapes(case):
            z, y, x = (torch.arange(m, dtype=torch.float64, device="cuda") for m in s)
            v = torch.zeros(s, dtype=torch.float64, device="cuda")
            for _ in range(4):
                k = (2 * math.pi * torch.rand(3, generator=g, dtype=torch.float64)).tolist()
                p = (2 * math.pi * torch.rand(3, generator=g, dtype=torch.float64)).tolist()
                v += (torch.cos(k[0] * x / n[0] + p[0])[None, None, :] * torch.cos(k[1] * y / n[1] + p[1])[None, :, None]
                      * torch.cos(k[2] * z / n[2] + p[2])[:, None, None])
            noise = torch.rand(s, generator=torch.Generator("cuda").manual_seed(int(torch.randint(1 << 30, (1,), generator=g))),
                               dtype=torch.float64, device="cuda")
            parts.append((v + 0.02 * (noise - 0.5)).reshape(-1))
        out.append(torch.cat(parts))
    return torch.stack(out) if count > 1 else out[0]


def _inputs(case, seed):
    """The level set(s), and what else the call reads."""
    g = _gen(seed)
    if case["call"] == "batch":
        jobs = []
        for i in range(case["count"]):
            n = (32, 48, 32, 64, 48, 32)[i]
            c = dict(case, shape=("sphere", "ellipsoid")[i % 2], nx=n, ny=n, nz=n)
            jobs.append((c, _phi(c, g), 2.0 + 4.0 * float(torch.rand(1, generator=g)), 4 + (i + case["nev"]) % 4))
        return {"jobs": jobs}
    d = {"phi": _phi(case, g)}
    if case["call"] != "modes":
        A = _fractions(d["phi"])[1] if case["call"] in ("solve", "certify", "train") else None
        x = _field(case, g, case["nev"] if case["call"] == "certify" else 1)
        if case["call"] == "certify" and case["nev"] == 1:
            x = x[None]
        if case["call"] == "certify":
            x *= (A > 0)
            d["k2"] = (7.0 + 20.0 * torch.rand(case["nev"], generator=g, dtype=torch.float64)).tolist()
        # a solve's right-hand side is A times a field; a residual to train on vanishes on closed faces
        d["x"] = A * x if case["call"] in ("solve", "train") else x
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    ctx = dm.Context(0)
    s = {"case": case, "ctx": ctx, **d}

    def geometry(c, phi):
        return dm.Geometry(ctx, c["nx"], c["ny"], c["nz"], *_spacing(c), phi.reshape(-1))

    if case["call"] == "batch":
        # the level sets of a sweep stay; the geometries are made once for it
        s["geoms"] = [geometry(c, phi) for c, phi, _, _ in d["jobs"]]
        return s
    if case["call"] != "modes":
        s["geom"] = geometry(case, d["phi"])
        if case["call"] != "certify":
            s["op"] = dm.Operator(ctx, s["geom"], _sigma(case), precision=case["precision"])
    if case["call"] == "train":
        s["net"] = dm.Learned(ctx, seed=int(seed) & 0xFFFF)
    if case["call"] == "apply_noalloc":
        s["out"] = torch.empty_like(d["x"])
    return s


def run(s):
    case, call = s["case"], s["case"]["call"]
    if call == "apply_noalloc":
        return s["op"].apply_noalloc(s["x"], out=s["out"])
    if call == "apply":
        return s["op"].apply(s["x"])
    if call == "certify":
        return list(dm.certify(s["ctx"], s["geom"], s["k2"], s["x"]))
    if call == "project":
        return s["op"].project(s["x"])[0]
    if call == "solve":
        return s["op"].solve(s["x"])[0]
    if call == "train":
        return list(s["net"].train_step(s["op"], s["x"], lr=1e-3))
    if call == "modes":
        geom = dm.Geometry(s["ctx"], case["nx"], case["ny"], case["nz"], *_spacing(case), s["phi"].reshape(-1))
        return dm.eigensolve(s["ctx"], geom, case["sigma"], case["nev"], vectors=None, precision=case["precision"])[0]
    jobs = [{"geom": g, "sigma": j[2], "nev": j[3], "precision": case["precision"]} for g, j in zip(s["geoms"], s["jobs"])]
    return [r[0] for r in dm.eigensolve_batched(s["ctx"], jobs)]


def work(case):
    """Inputs and fractions read once, results written once, in FP64; the flops of the products these calls are made of."""
    if case["call"] == "batch":
        cells = sum(n ** 3 for n in (32, 48, 32, 64, 48, 32)[:case["count"]])
        return {"bytes": 8.0 * cells, "flops": 100.0 * 3 * cells * (4 + case["nev"])}
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    faces = sum(a * b * c for a, b, c in _shapes(case))
    cells, nodes = nx * ny * nz, (nx + 1) * (ny + 1) * (nz + 1)
    fractions = 8.0 * (2 * faces + cells)
    if case["call"] == "modes":
        return {"bytes": 8.0 * nodes, "flops": 100.0 * faces * case["nev"]}
    if case["call"] == "train":   # three layers of 27 taps (8-16-16-3), forward, backward and weight gradients
        return {"bytes": 8.0 * faces + fractions, "flops": 3 * 2.0 * 27 * (8 * 16 + 16 * 16 + 16 * 3) * nodes}
    n = case["nev"] if case["call"] == "certify" else 1
    out = 0.0 if case["call"] == "certify" else 8.0 * faces
    return {"bytes": n * 8.0 * faces + out + fractions, "flops": 50.0 * faces * n}


# ---- what the outputs are in 64 bits, by plain torch ---------------------------------------------------------------

def _part(*v):
    """The part of a simplex (segment, triangle, tetrahedron) on whose corners the linear function takes the values v
    where that function is negative."""
    q = torch.sort(torch.stack(torch.broadcast_tensors(*v)), dim=0).values
    neg, m = (q < 0).sum(0), len(v) - 1

    def cut(a, others):   # the corner at a, of the other sign than the others
        r = torch.ones_like(q[0])
        for b in others:
            r = r * (q[a] / (q[a] - q[b]))
        return r

    out = (neg == m + 1).to(q.dtype)
    out = torch.where(neg == 1, cut(0, range(1, m + 1)), out)
    if m >= 2:
        out = torch.where(neg == m, 1.0 - cut(m, range(m)), out)
    if m == 3:   # two and two: a prism, as three tetrahedra
        al, be, ga, de = q[0] / (q[0] - q[2]), q[0] / (q[0] - q[3]), q[1] / (q[1] - q[2]), q[1] / (q[1] - q[3])
        out = torch.where(neg == 2, al * be * (1 - de) + al * de * (1 - ga) + ga * de, out)
    return out


def _fractions(phi):
    """Edge, face and cell fractions in natural layouts (conducting outer walls)."""
    p, L, A = phi, [], []
    nz, ny, nx = (s - 1 for s in p.shape)
    for axis in range(3):   # x, y, z
        d = 2 - axis
        e = _part(p.narrow(d, 0, p.shape[d] - 1), p.narrow(d, 1, p.shape[d] - 1))
        u, w = [2 - a for a in range(3) if a != axis]
        for dim in (u, w):   # tangential edges of the walls
            e.select(dim, 0).zero_()
            e.select(dim, e.shape[dim] - 1).zero_()
        L.append(e.reshape(-1))
        c = {(i, j): p.narrow(u, i, p.shape[u] - 1).narrow(w, j, p.shape[w] - 1) for i in (0, 1) for j in (0, 1)}
        f = 0.5 * (_part(c[0, 0], c[1, 0], c[1, 1]) + _part(c[0, 0], c[0, 1], c[1, 1]))
        f.select(d, 0).zero_()
        f.select(d, f.shape[d] - 1).zero_()
        A.append(f.reshape(-1))

    def corner(x, y, z):
        return p[z:z + nz, y:y + ny, x:x + nx]

    V = 0.0
    for a, b in ((0, 1), (0, 2), (1, 0), (1, 2), (2, 0), (2, 1)):
        s, t = [0, 0, 0], [0, 0, 0]
        s[a] = t[a] = t[b] = 1
        V = V + _part(corner(0, 0, 0), corner(*s), corner(*t), corner(1, 1, 1))
    return torch.cat(L), torch.cat(A), (V / 6.0).reshape(-1)


class _Ops:
    """C L C^T, A D^T V^-1 D A and D A D^T on natural arrays."""

    def __init__(self, case, phi):
        self.case, self.h = case, _spacing(case)
        L, self.A, V = _fractions(phi)
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        es = (nz + 1, ny + 1, nx), (nz + 1, ny, nx + 1), (nz, ny + 1, nx + 1)
        self.L = [v.reshape(s) for v, s in zip(torch.split(L, [math.prod(s) for s in es]), es)]
        self.V = V.reshape(nz, ny, nx)
        self.iV = torch.where(self.V > 0, 1.0 / self.V, torch.zeros_like(self.V))

    def split(self, x):
        s = _shapes(self.case)
        return [v.reshape(t) for v, t in zip(torch.split(x, [math.prod(t) for t in s]), s)]

    def div(self, x):
        fx, fy, fz = self.split(x)
        return ((fx[:, :, 1:] - fx[:, :, :-1]) / self.h[0] + (fy[:, 1:] - fy[:, :-1]) / self.h[1]
                + (fz[1:] - fz[:-1]) / self.h[2])

    def grad(self, p):   # D^T, closed walls
        out = []
        for s, d, h in zip(_shapes(self.case), (2, 1, 0), self.h):
            g = torch.zeros(s, dtype=p.dtype, device=p.device)
            g.narrow(d, 1, s[d] - 2).copy_((p.narrow(d, 0, s[d] - 2) - p.narrow(d, 1, s[d] - 2)) / h)
            out.append(g.reshape(-1))
        return torch.cat(out)

    def K(self, b, sigma):
        bx, by, bz = self.split(b)
        dx, dy, dz = self.h
        ex, ey, ez = (torch.zeros_like(v) for v in self.L)
        ex[1:-1, 1:-1] = (by[:-1, 1:-1] - by[1:, 1:-1]) / dz + (bz[1:-1, 1:] - bz[1:-1, :-1]) / dy
        ey[1:-1, :, 1:-1] = (bx[1:, :, 1:-1] - bx[:-1, :, 1:-1]) / dz + (bz[1:-1, :, :-1] - bz[1:-1, :, 1:]) / dx
        ez[:, 1:-1, 1:-1] = (bx[:, :-1, 1:-1] - bx[:, 1:, 1:-1]) / dy + (by[:, 1:-1, 1:] - by[:, 1:-1, :-1]) / dx
        ex, ey, ez = ex * self.L[0], ey * self.L[1], ez * self.L[2]
        cx = (ez[:, 1:] - ez[:, :-1]) / dy - (ey[1:] - ey[:-1]) / dz
        cy = (ex[1:] - ex[:-1]) / dz - (ez[:, :, 1:] - ez[:, :, :-1]) / dx
        cz = (ey[:, :, 1:] - ey[:, :, :-1]) / dx - (ex[:, 1:] - ex[:, :-1]) / dy
        curl = torch.cat([cx.reshape(-1), cy.reshape(-1), cz.reshape(-1)])
        y = curl + self.A * (self.grad(self.iV * self.div(self.A * b)) - sigma * b)
        return torch.where(self.A > 0, y, torch.zeros_like(y))

    def diag(self, sigma):
        rx, ry, rz = (1.0 / h ** 2 for h in self.h)
        lx, ly, lz = self.L
        ax, ay, az = self.split(self.A)

        def two(d):   # V^-1 of the two cells of each face
            z = torch.zeros_like(self.iV.narrow(d, 0, 1))
            return torch.cat([z, self.iV], d) + torch.cat([self.iV, z], d)

        dx = (lz[:, :-1] + lz[:, 1:]) * ry + (ly[:-1] + ly[1:]) * rz + ax ** 2 * two(2) * rx - sigma * ax
        dy = (lx[:-1] + lx[1:]) * rz + (lz[:, :, :-1] + lz[:, :, 1:]) * rx + ay ** 2 * two(1) * ry - sigma * ay
        dz = (ly[:, :, :-1] + ly[:, :, 1:]) * rx + (lx[:, :-1] + lx[:, 1:]) * ry + az ** 2 * two(0) * rz - sigma * az
        d = torch.cat([dx.reshape(-1), dy.reshape(-1), dz.reshape(-1)])
        return torch.where(self.A > 0, d, torch.ones_like(d))


def _conjugate(mul, diag, b, rel, most, restarts=4):
    """mul^-1 b by diagonally preconditioned conjugate gradients, each restart on the true residual; None if it stalls."""
    x, goal = torch.zeros_like(b), rel * float(b.norm())
    for _ in range(restarts):
        r = b - mul(x)
        if float(r.norm()) <= goal:
            return x
        z = r / diag
        p, rz = z.clone(), torch.dot(r, z)
        for i in range(most):
            q = mul(p)
            a = rz / torch.dot(p, q)
            x = x + a * p
            r = r - a * q
            if i % 25 == 0 and float(r.norm()) <= 0.3 * goal:
                break
            z = r / diag
            new = torch.dot(r, z)
            p = z + (new / rz) * p
            rz = new
    return x if float((b - mul(x)).norm()) <= 1e-12 * float(b.norm()) else None


def exact(case, seed):
    call, faces = case["call"], sum(math.prod(s) for s in _shapes(case))
    # a whole batch, the trained network's BF16 layers, and solves of millions of unknowns take minutes in 64 bits
    if call in ("batch", "train") or (call == "solve" and faces > 1_500_000) or (call == "modes" and faces > 14_000):
        return None
    d = _inputs(case, seed)
    ops = _Ops(case, d["phi"])
    A, h = ops.A, ops.h
    inside = A > 0
    if call in ("apply", "apply_noalloc"):
        return ops.K(torch.where(inside, d["x"], torch.zeros_like(d["x"])), _sigma(case))
    if call == "certify":
        rho, delta, rq = [], [], []
        for k2, b in zip(d["k2"], d["x"]):
            kb, ab = ops.K(b, 0.0), A * b
            rq.append(torch.dot(b, kb) / torch.dot(b, ab))
            rho.append((kb - k2 * ab).norm() / (k2 * ab.norm()))
            delta.append(ops.div(ab).norm() * min(h) / ab.norm())
        return [torch.stack(v) for v in (rho, delta, rq)]
    if call == "project":
        x = torch.where(inside, d["x"], torch.zeros_like(d["x"]))
        s = ops.div(A * x)
        live = ops.V > 0
        ax, ay, az = ops.split(A)
        diag = ((ax[:, :, 1:] + ax[:, :, :-1]) / h[0] ** 2 + (ay[:, 1:] + ay[:, :-1]) / h[1] ** 2
                + (az[1:] + az[:-1]) / h[2] ** 2)
        diag = torch.where(live & (diag > 0), diag, torch.ones_like(diag))
        shape = s.shape
        psi = _conjugate(lambda v: ops.div(A * ops.grad(v.reshape(shape))).reshape(-1), diag.reshape(-1),
                         s.reshape(-1), 1e-14, 6000)
        return None if psi is None else torch.where(inside, x - ops.grad(psi.reshape(shape)), torch.zeros_like(x))
    if call == "solve":
        return _conjugate(lambda v: ops.K(v, _sigma(case)), ops.diag(_sigma(case)), d["x"], 1e-14, 8000)
    # modes: block inverse iteration on the dense matrix, whose grad-div part is weighted so that the divergent modes
    # leave the neighbourhood of the shift, then Rayleigh quotients of C L C^T
    idx = torch.nonzero(inside).reshape(-1)
    n, nev = idx.numel(), case["nev"]
    M0, M1 = (torch.empty(n, n, dtype=torch.float64, device="cuda") for _ in range(2))
    e = torch.zeros_like(A)
    for j in range(n):
        e[idx[j]] = 1.0
        gd = torch.where(inside, A * ops.grad(ops.iV * ops.div(A * e)), torch.zeros_like(A))
        M1[:, j] = gd[idx]
        M0[:, j] = ops.K(e, 0.0)[idx] - M1[:, j]
        e[idx[j]] = 0.0
    a = A[idx]
    lu = torch.linalg.lu_factor(M0 + 100.0 * M1 - torch.diag(case["sigma"] * a))
    X = torch.rand(n, 4 * nev + 8, generator=torch.Generator("cuda").manual_seed(1), dtype=torch.float64, device="cuda")
    for _ in range(40):
        X = torch.linalg.qr(torch.linalg.lu_solve(*lu, a[:, None] * X))[0]
    C = torch.linalg.cholesky(X.T @ (a[:, None] * X))
    X = torch.linalg.solve_triangular(C, X.T, upper=False).T
    w, U = torch.linalg.eigh(X.T @ (M0 @ X))
    div = torch.stack([ops.div(A * torch.zeros_like(A).index_copy(0, idx, v)).norm() for v in (X @ U).T])
    w = w[div < 1e-3 * w.abs().clamp(min=1.0)]
    return torch.sort(w[torch.argsort((w - case["sigma"]).abs())[:nev]]).values
