"""What the framework is used for, as measurable cases.

A case is one call, or one short sequence of calls, that a user's program makes
through the public binding (`paper_1704_02745_gb300.pb`):

  apply      the operator on a vector (a program's own solver or residual check)
  step       one MD snapshot: new atoms into a resident grid, a solve that
             starts from the previous snapshot's potential, the energy
  solve      a solve from zero on a grid that is set up, and the energy
  solvation  the solvation energy: two systems, each set up and solved
  serve      a burst of snapshots through the continuous-batching server

Atoms are the package's seeded globules.  A program that asks for 1e-6 writes
its potential map in single precision, and so do the cases here; tighter
solves return the FP64 potential itself.

`exact` restates the model (dielectric, charges, Debye-Hueckel boundary,
seven-point operator) in FP64 torch and solves it to 1e-12.
"""
import math

import numpy as np
import torch

from paper_1704_02745_gb300 import inputs, pb

ENERGY_UNIT = 332.0637  # kcal/mol per e^2/A
MB = 1 << 20

# ---------------------------------------------------------------------------
# The cases.  h and radius place the grid: nodes h apart, atoms in a ball.

_BASE = {"kind": "solve", "nx": 129, "ny": 129, "nz": 129, "h": 0.5, "radius": 24.0, "atoms": 2500,
         "coef": "packed", "dh": "f32", "periodic": False, "eps_model": "midpoint",
         "precision": "f32_refine", "precond": "jacobi", "tol": 1e-6, "inner_tol": 1e-4, "count": 1}


def _case(**kw):
    c = dict(_BASE)
    c.update(kw)
    if "n" in c:
        c["nx"] = c["ny"] = c["nz"] = c.pop("n")
    return c


def listed():
    return [
        # the smallest call: one operator application, all latency
        _case(name="apply_33", kind="apply", n=33, radius=7.0, atoms=200, precision="f64", dh="f64"),
        # a small solute's snapshot in an MD loop
        _case(name="step_33", kind="step", n=33, radius=7.0, atoms=200),
        # the ordinary protein-sized snapshot
        _case(name="step_129", kind="step", n=129),
        # the largest solute of a served stream, a box that is not a cube
        _case(name="step_187x161x175", kind="step", nx=187, ny=161, nz=175, h=0.61, radius=30.0, atoms=5400),
        # a large complex, one-byte coefficients
        _case(name="solve_257", n=257, radius=50.0, atoms=20000),
        # the same complex with explicit BF16 coefficients, refined to 1e-9
        _case(name="solve_257_bf16", n=257, radius=50.0, atoms=20000, coef="bf16", tol=1e-9, inner_tol=1e-3),
        # the published method in FP64 throughout
        _case(name="solve_129_f64", n=129, precision="f64", dh="f64"),
        # the multigrid preconditioner
        _case(name="solve_129_gmg", n=129, precision="f64", precond="gmg", dh="f64"),
        # a periodic box
        _case(name="step_periodic", kind="step", nx=97, ny=81, nz=113, h=0.6, radius=16.0, atoms=690,
              periodic=True, tol=1e-9),
        # the weighted harmonic-average dielectric (FP32 copies of FP64 edges)
        _case(name="step_harmonic_97", kind="step", n=97, h=0.5, radius=18.0, atoms=1000, coef="f32",
              eps_model="harmonic", tol=1e-9, inner_tol=1e-3),
        # a solvation energy with every default of the grid (FP64 boundary sum)
        _case(name="solvation_97", kind="solvation", n=97, h=0.5, radius=18.0, atoms=1000, dh="f64"),
        # a burst of one cluster's snapshots on grids of 49 to 97 nodes a side
        _case(name="serve_32", kind="serve", n=97, h=0.0, radius=18.0, atoms=1000, count=32, tol=1e-9),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _ball(nmin, h):
    """Radius and atom count that leave the grid 1.5 times the solute's extent."""
    radius = max(4.0, (h * (nmin - 1) / inputs.FILL_RATIO - 2 * inputs.R_MAX) / 2)
    return round(radius, 2), max(20, int(inputs.ATOM_DENSITY * 4 / 3 * math.pi * radius ** 3))


def draw(rng):
    kind = rng.choice(["apply", "step", "step", "step", "solve", "solve", "solvation", "serve"])
    if kind == "serve":
        return _case(kind="serve", n=_log_int(rng, 57, 97), h=0.0, radius=18.0, atoms=1000,
                     count=_log_int(rng, 4, 32), tol=1e-9)
    top = {"apply": 257, "step": 181, "solve": 225, "solvation": 97}[kind]
    n = _log_int(rng, 33, top)
    dims = [n, n, n]
    if rng.random() < 0.6:  # a box that is not a cube
        dims = [max(29, min(top, int(n * rng.uniform(0.8, 1.25)))) for _ in range(3)]
    h = round(rng.uniform(0.45, 0.75), 3)
    radius, atoms = _ball(min(dims), h)
    kw = dict(kind=kind, nx=dims[0], ny=dims[1], nz=dims[2], h=h, radius=radius, atoms=atoms)
    if kind == "apply":
        kw.update(precision=rng.choice(["f64", "f32"]), coef=rng.choice(["packed", "f32", "bf16"]))
    elif kind == "solvation":
        kw.update(dh=rng.choice(["f64", "f32"]))
    else:
        variant = rng.choice(["packed", "packed", "f32", "bf16", "f64", "gmg", "periodic", "harmonic"])
        if variant == "f32" or variant == "bf16":
            kw.update(coef=variant, tol=1e-9, inner_tol=1e-3)
        elif variant in ("f64", "gmg"):
            # FP64 arithmetic: a pass of the largest costs what the largest listed case does
            dims = [min(d, 161) for d in dims]
            kw.update(nx=dims[0], ny=dims[1], nz=dims[2], precision="f64",
                      precond="gmg" if variant == "gmg" else "jacobi")
            kw["radius"], kw["atoms"] = _ball(min(dims), h)
        elif variant == "periodic":
            kw.update(periodic=True, tol=1e-9)
        elif variant == "harmonic":
            kw.update(coef=rng.choice(["f32", "bf16"]), eps_model="harmonic", tol=1e-9, inner_tol=1e-3)
            if max(dims) > 129:
                dims = [min(d, 129) for d in dims]
                kw.update(nx=dims[0], ny=dims[1], nz=dims[2])
                kw["radius"], kw["atoms"] = _ball(min(dims), h)
    return _case(**kw)


# ---------------------------------------------------------------------------
# Problems from a case and a seed (host arrays; no arithmetic of the method)

def _spec(c, n=None):
    nx, ny, nz = (n, n, n) if n else (c["nx"], c["ny"], c["nz"])
    h = c["h"] or inputs.fill_spacing(n, c["radius"])
    origin = tuple(-h * (m - 1) / 2.0 for m in (nx, ny, nz))
    return inputs.GridSpec(nx, ny, nz, h, origin, coef=c["coef"], dh=c["dh"], periodic=c["periodic"],
                           eps_model=c["eps_model"])


def _snapshots(c, seed, count, sigma):
    """One globule and `count` perturbed copies of it."""
    rng = np.random.default_rng([seed, 11])
    base = inputs.ball_atoms(rng, c["atoms"], c["radius"])
    out = [base]
    for _ in range(count):
        a = base.copy()
        a.xyz = a.xyz + rng.normal(0.0, sigma, size=a.xyz.shape)
        out.append(a)
    return out


def _burst(c, seed):
    """The served burst: (grid, atoms) of each request, 49 .. nx nodes a side."""
    snaps = _snapshots(c, seed, c["count"], 0.3)[1:]
    sizes = np.random.default_rng([c["nx"], c["count"]]).integers(49, c["nx"] + 1, c["count"])
    return [(_spec(c, int(n)), a) for n, a in zip(sizes, snaps)]


# ---------------------------------------------------------------------------
# What a program holds, and one pass

_program = {}


def _context():
    """The program's stream and its context on it."""
    if not _program:
        _program["stream"] = torch.cuda.Stream()
        _program["ctx"] = pb.Context(0, stream=_program["stream"].cuda_stream)
    return _program["ctx"], _program["stream"]


class State:
    def __init__(self, **kw):
        self.__dict__.update(kw)

    def __del__(self):
        for k in ("grid", "server"):
            if getattr(self, k, None) is not None:
                getattr(self, k).close()


def _options(c):
    return dict(precision=c["precision"], precond=c["precond"], tol=c["tol"], inner_tol=c["inner_tol"])


def prepare(case, seed):
    ctx, stream = _context()
    s = State(kind=case["kind"], case=case, stream=stream, ctx=ctx, opts=_options(case),
              single=case["tol"] >= 1e-6 and case["precision"] != "f64")
    if case["kind"] == "serve":
        s.requests = _burst(case, seed)
        s.out = [pb.pinned_empty(tuple(g.shape)) for g, _ in s.requests]
        s.server = pb.Server(ctx, 16384 * MB, warm_start=False, **s.opts)
        return s
    spec = _spec(case)
    before, atoms = _snapshots(case, seed, 1, 0.2)
    s.spec, s.atoms = spec, atoms
    with torch.cuda.stream(stream):
        if case["kind"] == "apply":
            g = torch.Generator(device="cuda")
            g.manual_seed(int(seed))
            dt = torch.float64 if case["precision"] == "f64" else torch.float32
            s.u = torch.randn(spec.shape, generator=g, dtype=dt, device="cuda")
            s.au = torch.empty_like(s.u)
            s.dtype = pb.PB_F64 if case["precision"] == "f64" else pb.PB_F32
            s.grid = pb.Grid(ctx, spec, atoms)
            return s
        s.phi = torch.zeros(spec.shape, dtype=torch.float64, device="cuda")
        if case["kind"] == "step":  # the previous snapshot, solved
            s.grid = pb.Grid(ctx, spec, before)
            s.grid.solve(s.phi, **s.opts)
            s.before = s.phi.clone()
        elif case["kind"] == "solve":
            s.grid = pb.Grid(ctx, spec, atoms)
    stream.synchronize()
    return s


def run(state):
    s = state
    if s.kind == "serve":
        tickets = [s.server.submit(k, g, a, phi_out=o) for k, ((g, a), o) in enumerate(zip(s.requests, s.out))]
        results = [s.server.poll(t) for t in tickets]
        return {"energy": np.array([r.energy for r, _ in results]), "phi": [phi for _, phi in results]}
    with torch.cuda.stream(s.stream):
        if s.kind == "apply":
            s.grid.apply(s.u, s.au, s.dtype)
            return s.au
        if s.kind == "solvation":
            r = s.ctx.solvation(s.spec, s.atoms, s.phi, **s.opts)
            return {"phi": s.phi.float() if s.single else s.phi, "dG": r.dG, "e_solv": r.e_solv, "e_ref": r.e_ref}
        if s.kind == "step":
            s.phi.copy_(s.before)
            s.grid.update_atoms(s.atoms)
        s.grid.solve(s.phi, warm_start=s.kind == "step", **s.opts)
        energy = s.grid.energy(s.phi)
        return {"phi": s.phi.float() if s.single else s.phi, "energy": energy}


# ---------------------------------------------------------------------------
# The work a pass cannot do without: inputs read once, outputs written once,
# and the operations of the conjugate-gradient iterations such a grid takes
# (27 a node: two fused updates, seven products, two dot products).

def _iterations(c, nmax):
    per_digit = 5.0 if c["precond"] == "gmg" else 0.12 * nmax + 18.0
    return per_digit * -math.log10(c["tol"])


def work(case):
    c = case
    if c["kind"] == "serve":
        dims = [(m, m, m) for m in np.linspace(49, c["nx"], c["count"])]
    else:
        dims = [(c["nx"], c["ny"], c["nz"])]
    n = float(sum(a * b * d for a, b, d in dims))
    if c["kind"] == "apply":
        return {"bytes": n * (17 if c["precision"] == "f64" else 9), "flops": 13 * n}
    systems = 2 if c["kind"] == "solvation" else 1
    nbytes = n * 8 * (2 if c["kind"] == "step" else 1) + 40.0 * c["atoms"] * c["count"]
    pairs = 0.0 if c["periodic"] else sum(2 * (a * b + b * d + a * d) for a, b, d in dims) * c["atoms"]
    if c["kind"] == "solve":
        pairs = 0.0
    return {"bytes": nbytes, "flops": systems * (27 * n * _iterations(c, max(max(d) for d in dims)) + 12 * pairs)}


# ---------------------------------------------------------------------------
# The model in FP64, in plain torch

_F = torch.float64


def _axis(o, count, h, shift):
    """Coordinates o + (i + shift) * h of `count` lattice points."""
    return o + (torch.arange(count, device="cuda", dtype=_F) + shift) * h


def _inside(spec, atoms, first, dims, shift):
    """True where lattice point (x, y, z), at index first + i shifted by
    `shift` spacings, lies strictly inside an atom (or, on a periodic grid, one
    of its images; `dims` then is the period)."""
    h, o = spec.h, spec.origin
    flag = torch.zeros(dims[2] * dims[1] * dims[0], dtype=torch.bool, device="cuda")
    xyz = torch.as_tensor(atoms.xyz, device="cuda")
    rad = torch.as_tensor(atoms.r, device="cuda")
    m = int(math.ceil(2 * float(atoms.r.max()) / h)) + 4
    off = torch.arange(m, device="cuda")
    step = max(1, 20_000_000 // m ** 3)
    for a in range(0, atoms.n, step):
        p, r = xyz[a:a + step], rad[a:a + step]
        idx, d2, ok = [], [], []
        for ax in range(3):
            i = torch.floor((p[:, ax] - r - o[ax]) / h - shift[ax]).long()[:, None] - 1 + off
            c = o[ax] + (i.to(_F) + shift[ax]) * h
            d2.append((c - p[:, ax, None]) ** 2)
            i = i - first[ax]
            ok.append(torch.ones_like(i, dtype=torch.bool) if spec.periodic else (i >= 0) & (i < dims[ax]))
            idx.append(i.remainder(dims[ax]))
        dist = (d2[0][:, None, None, :] + d2[1][:, None, :, None]) + d2[2][:, :, None, None]
        hit = (dist < (r * r)[:, None, None, None]) & ok[0][:, None, None, :] & ok[1][:, None, :, None] \
            & ok[2][:, :, None, None]
        flat = (idx[2][:, :, None, None] * dims[1] + idx[1][:, None, :, None]) * dims[0] + idx[0][:, None, None, :]
        flag[flat[hit]] = True
    return flag.view(dims[2], dims[1], dims[0])


def _covered(spec, atoms, ax, dims):
    """Fraction of each edge along `ax` (entry e: from node e-1 to node e)
    strictly inside the union of the atoms."""
    h, o = spec.h, spec.origin
    xyz = torch.as_tensor(atoms.xyz, device="cuda")
    rad = torch.as_tensor(atoms.r, device="cuda")
    m = int(math.ceil(2 * float(atoms.r.max()) / h)) + 4
    off = torch.arange(m, device="cuda")
    edges, los, his = [], [], []
    step = max(1, 10_000_000 // m ** 3)
    for a in range(0, atoms.n, step):
        p, r = xyz[a:a + step], rad[a:a + step]
        idx, pos, ok = [], [], []
        for d in range(3):
            i = torch.floor((p[:, d] - r - o[d]) / h).long()[:, None] - 1 + off
            pos.append(o[d] + i.to(_F) * h)
            e = i + 1 if d == ax else i
            ok.append((e >= 0) & (e < dims[d]))
            idx.append(e.clamp(0, dims[d] - 1))

        def lay(v, d):
            return v[:, None, None, :] if d == 0 else v[:, None, :, None] if d == 1 else v[:, :, None, None]

        u, v = [d for d in range(3) if d != ax]
        s = (r * r)[:, None, None, None] - (lay((pos[u] - p[:, u, None]) ** 2, u) + lay((pos[v] - p[:, v, None]) ** 2, v))
        q = torch.sqrt(s.clamp_min(0.0))
        rel = lay(p[:, ax, None] - pos[ax], ax)
        lo, hi = ((rel - q) / h).clamp_min(0.0), ((rel + q) / h).clamp_max(1.0)
        hit = (s > 0) & (lo < hi) & lay(ok[0], 0) & lay(ok[1], 1) & lay(ok[2], 2)
        flat = (lay(idx[2], 2) * dims[1] + lay(idx[1], 1)) * dims[0] + lay(idx[0], 0)
        edges.append(flat[hit])
        los.append(lo[hit])
        his.append(hi[hit])
    edge, lo, hi = torch.cat(edges), torch.cat(los), torch.cat(his)
    order = torch.argsort(lo, stable=True)
    order = order[torch.argsort(edge[order], stable=True)]
    edge, lo, hi = edge[order], lo[order], hi[order]
    n = dims[0] * dims[1] * dims[2]
    count = torch.bincount(edge, minlength=n)
    start = torch.cumsum(count, 0) - count
    rank = torch.arange(edge.numel(), device="cuda") - start[edge]
    w = torch.zeros(n, dtype=_F, device="cuda")
    end = torch.zeros(n, dtype=_F, device="cuda")  # right end of what is covered so far
    for k in range(int(count.max()) if edge.numel() else 0):
        at = rank == k
        e = edge[at]
        w[e] += (hi[at] - torch.maximum(lo[at], end[e])).clamp_min(0.0)
        end[e] = torch.maximum(end[e], hi[at])
    return w.clamp_max(1.0).view(dims[2], dims[1], dims[0])


class Model:
    """A phi = b of one system, FP64."""

    def __init__(self, spec, atoms):
        nx, ny, nz, h = spec.nx, spec.ny, spec.nz, spec.h
        self.spec, self.atoms, per = spec, atoms, spec.periodic
        ein, eout = spec.eps_in, spec.eps_out
        self.eps = []
        for ax in range(3):
            dims, first, shift = [nx, ny, nz], [0, 0, 0], [0.0, 0.0, 0.0]
            if spec.eps_model == "harmonic":
                dims[ax] += 1
                w = _covered(spec, atoms, ax, dims)
                self.eps.append(1.0 / (w / ein + (1.0 - w) / eout))
                continue
            shift[ax] = 0.5
            first[ax] = -1
            if not per:
                dims[ax] += 1
            e = torch.where(_inside(spec, atoms, first, dims, shift), ein, eout).to(_F)
            if per:  # entry n is entry 0
                e = torch.cat([e, e.narrow(2 - ax, 0, 1)], 2 - ax)
            self.eps.append(e)
        lam = torch.ones((nz, ny, nx), dtype=_F, device="cuda")
        if spec.kappa_mask:
            lam = 1.0 - _inside(spec, atoms, [0, 0, 0], [nx, ny, nz], [0.0, 0.0, 0.0]).to(_F)
        # Debye length: SI constants, lengths in A
        kappa2 = 2.0 * 6.02214076e23 * 1.602176634e-19 ** 2 * (1000.0 * spec.ionic_strength) / (
            8.8541878128e-12 * eout * 1.380649e-23 * spec.temperature) * 1e-20
        self.kappa = math.sqrt(kappa2)
        self.diag = lam * (eout * kappa2 * h * h)
        for ax in range(3):
            n = (nx, ny, nz)[ax]
            self.diag += self.eps[ax].narrow(2 - ax, 0, n) + self.eps[ax].narrow(2 - ax, 1, n)
        self.corners()
        self.b = torch.zeros(nz * ny * nx, dtype=_F, device="cuda")
        for at, w in self.at:
            self.b.index_add_(0, at, w * (4.0 * math.pi / h))
        self.b = self.b.view(nz, ny, nx)
        if not per:
            self.boundary()

    def corners(self):
        """(flat node, charge share) of the eight corners of each atom's cell."""
        s = self.spec
        xyz = torch.as_tensor(self.atoms.xyz, device="cuda")
        q = torch.as_tensor(self.atoms.q, device="cuda")
        n = (s.nx, s.ny, s.nz)
        f = [(xyz[:, d] - s.origin[d]) / s.h for d in range(3)]
        c = [torch.floor(v) for v in f]
        w = [(1.0 - (v - k), v - k) for v, k in zip(f, c)]
        self.at = []
        for dk in range(2):
            for dj in range(2):
                for di in range(2):
                    i, j, k = [(c[d].long() + (di, dj, dk)[d]) for d in range(3)]
                    if s.periodic:
                        i, j, k = i.remainder(n[0]), j.remainder(n[1]), k.remainder(n[2])
                    self.at.append(((k * n[1] + j) * n[0] + i, q * w[0][di] * w[1][dj] * w[2][dk]))

    def boundary(self):
        s = self.spec
        n = (s.nx, s.ny, s.nz)
        xyz = torch.as_tensor(self.atoms.xyz, device="cuda")
        q = torch.as_tensor(self.atoms.q, device="cuda") / s.eps_out
        for ax in range(3):
            u, v = [d for d in range(3) if d != ax]  # u varies fastest
            cu, cv = _axis(s.origin[u], n[u], s.h, 0.0), _axis(s.origin[v], n[v], s.h, 0.0)
            for side in range(2):
                level = s.origin[ax] + (n[ax] if side else -1) * s.h
                fu, fv = cu.repeat(n[v]), cv.repeat_interleave(n[u])
                face = torch.empty(n[u] * n[v], dtype=_F, device="cuda")
                step = max(1, 50_000_000 // max(1, self.atoms.n))
                for a in range(0, face.numel(), step):
                    d2 = (fu[a:a + step, None] - xyz[None, :, u]) ** 2
                    d2 += (fv[a:a + step, None] - xyz[None, :, v]) ** 2
                    d2 += (level - xyz[None, :, ax]) ** 2
                    r = d2.sqrt_()
                    face[a:a + step] = (torch.exp(r * -self.kappa) / r) @ q
                k = n[ax] if side else 0
                # (v, u) is the order of the array's remaining axes
                self.b.select(2 - ax, k - 1 if side else 0).add_(
                    self.eps[ax].select(2 - ax, k) * face.view(n[v], n[u]))

    def apply(self, x):
        out = self.diag * x
        for ax in range(3):
            d, n, e = 2 - ax, x.shape[2 - ax], self.eps[ax]
            if self.spec.periodic:
                out -= e.narrow(d, 0, n) * torch.roll(x, 1, d)
                out -= e.narrow(d, 1, n) * torch.roll(x, -1, d)
            elif n > 1:
                mid = e.narrow(d, 1, n - 1)
                out.narrow(d, 1, n - 1).addcmul_(mid, x.narrow(d, 0, n - 1), value=-1.0)
                out.narrow(d, 0, n - 1).addcmul_(mid, x.narrow(d, 1, n - 1), value=-1.0)
        return out

    def solve(self, tol=1e-12, most=6000):
        x = torch.zeros_like(self.b)
        r = self.b.clone()
        stop = float(r.norm()) * tol
        z = r / self.diag
        p, rz = z.clone(), torch.sum(r * z)
        for it in range(most):
            ap = self.apply(p)
            alpha = rz / torch.sum(p * ap)
            x.addcmul_(p, alpha)
            r.addcmul_(ap, -alpha)
            if it % 10 == 9 and float(r.norm()) < stop:
                break
            z = r / self.diag
            new = torch.sum(r * z)
            p.mul_(new / rz).add_(z)
            rz = new
        return x

    def energy(self, x):
        flat = x.reshape(-1)
        return 0.5 * ENERGY_UNIT * float(sum(torch.sum(w * flat[at]) for at, w in self.at))


def exact(case, seed):
    if case["kind"] == "serve":
        energies, phis = [], []
        for spec, atoms in _burst(case, seed):
            m = Model(spec, atoms)
            x = m.solve()
            energies.append(m.energy(x))
            phis.append(x.cpu().numpy())
        return {"energy": np.array(energies), "phi": phis}
    spec = _spec(case)
    _, atoms = _snapshots(case, seed, 1, 0.2)
    if case["kind"] == "apply":
        g = torch.Generator(device="cuda")
        g.manual_seed(int(seed))
        dt = torch.float64 if case["precision"] == "f64" else torch.float32
        return Model(spec, atoms).apply(torch.randn(spec.shape, generator=g, dtype=dt, device="cuda").to(_F))
    m = Model(spec, atoms)
    x = m.solve()
    e = m.energy(x)
    if case["kind"] == "solvation":
        ref = Model(spec.replace(eps_out=spec.eps_in, ionic_strength=0.0), atoms)
        e_ref = ref.energy(ref.solve())
        return {"phi": x, "dG": e - e_ref, "e_solv": e, "e_ref": e_ref}
    return {"phi": x, "energy": e}
