"""Workloads for timing this framework through its public Python API.

Each case is a dict of plain values.  ``prepare`` builds what a user's program
holds before the call (device arrays, a context, its weights, a batch, a
network); ``run`` makes one pass through the public entry points and returns
its whole outputs; ``exact`` computes the same outputs in 64 bits with plain
torch operations, for the cases where that is affordable.

Kinds of case
  step2d   one implicit step on a 2D grid: weight build, then the solve to a
           true relative residual (``shape``: disk, or the sum of Gaussian
           bumps with a moving disk); what a simulation does every time step
  jet2d    one Navier-Stokes step of the planar jet: transport, weight build,
           Schwarz-preconditioned solve
  step3d   one implicit step of the 3D liquid column, as step2d
  batch    many uneven 2D instances solved in one persistent launch
  apply    one matrix-free apply y = A x (2D or 3D, FP64 / FP32 / BF16
           coefficients), for callers that run their own Krylov method
  net      the preconditioner network: inference on a whole grid, or one
           gradient of a training batch

Solves run to 1e-12: at that tolerance the returned velocities, stresses and
pressures are determined to about 1e-10, which is what a user who compares
two runs, or checks against a direct solve, asks for.
"""
import math

import numpy as np
import torch

from paper_1010_2832_gb300 import stokes

F64 = torch.float64
FLOOR = 0.01       # floor of the live faces' mass fraction, as the jet driver sets it


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest whole call: 32^2 liquid disk, plain FP64 PCG (latency of the CG loop)
        dict(name="step2d_disk32_fp64", kind="step2d", shape="disk", nx=32, ny=32, geom=1, precision=0, precond=0),
        # one time step of the planar jet driver at the size its study runs at
        dict(name="jet2d_150", kind="jet2d", n=150, geom=1),
        # the headline workload: 1024^2 bumps, FP32 Schwarz-CG inside FP64 refinement
        dict(name="step2d_bumps1024_mixed", kind="step2d", shape="bumps", nx=1024, ny=1024, geom=2, precision=1,
             precond=2),
        # a 3D step: thin liquid column in a large grid (weight build and a short Jacobi-PCG solve)
        dict(name="step3d_column256_mixed", kind="step3d", nx=256, ny=256, nz=256, precision=1),
        # the batched form: 12 uneven instances, FP64 PCG with the Schwarz preconditioner
        dict(name="batch12_fp64", kind="batch", count=12, lo=64, hi=160, geom=4000, precond=2),
        # applies over the range of sizes: roofline size, an FP64 one with an interface, a small ragged one
        dict(name="apply2d_box4096_fp32", kind="apply", dim=2, nx=4096, ny=4096, nz=0, shape="box", geom=0,
             precision=1),
        dict(name="apply2d_bumps1024_fp64", kind="apply", dim=2, nx=1024, ny=1024, nz=0, shape="bumps", geom=2,
             precision=0),
        dict(name="apply2d_bumps301x515_bf16", kind="apply", dim=2, nx=301, ny=515, nz=0, shape="bumps", geom=3,
             precision=2),
        dict(name="apply3d_box256_fp32", kind="apply", dim=3, nx=256, ny=256, nz=256, shape="box", geom=0,
             precision=1),
        dict(name="apply3d_bumps129x97x65_fp64", kind="apply", dim=3, nx=129, ny=97, nz=65, shape="bumps", geom=5,
             precision=0),
        # the network on a whole 3D grid (one preconditioner application) and on a training batch of windows
        dict(name="net3d_forward128", kind="net", dim=3, grad=False, B=1, D=128, H=128, W=128),
        dict(name="net3d_gradient4x64", kind="net", dim=3, grad=True, B=4, D=64, H=64, W=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "step2d", "step2d", "jet2d", "step3d", "batch", "net", "net"])
    geom = rng.randrange(1, 1000)
    if kind == "apply":
        dim = rng.choice([2, 3])
        lo, hi = (32, 4096) if dim == 2 else (16, 256)
        return dict(kind=kind, dim=dim, nx=_log_int(rng, lo, hi), ny=_log_int(rng, lo, hi),
                    nz=_log_int(rng, lo, hi) if dim == 3 else 0, shape=rng.choice(["box", "bumps"]), geom=geom,
                    precision=rng.choice([0, 1, 2]))
    if kind == "step2d":
        if rng.random() < 0.4:
            return dict(kind=kind, shape="disk", nx=_log_int(rng, 24, 128), ny=_log_int(rng, 24, 128), geom=geom,
                        precision=rng.choice([0, 1]), precond=rng.choice([0, 2]))
        n = _log_int(rng, 64, 640)
        return dict(kind=kind, shape="bumps", nx=n, ny=max(64, n - rng.randrange(0, n // 4)), geom=geom, precision=1,
                    precond=2)
    if kind == "jet2d":
        return dict(kind=kind, n=_log_int(rng, 100, 300), geom=geom)
    if kind == "step3d":
        return dict(kind=kind, nx=_log_int(rng, 64, 240), ny=_log_int(rng, 64, 240), nz=_log_int(rng, 64, 240),
                    precision=rng.choice([0, 1, 2]))
    if kind == "batch":
        lo = _log_int(rng, 48, 96)
        return dict(kind=kind, count=rng.randrange(3, 13), lo=lo, hi=lo + rng.randrange(10, 60), geom=geom, precond=2)
    if rng.random() < 0.5:
        dim = rng.choice([2, 3])
        hi = 24 if dim == 3 else 96
        return dict(kind=kind, dim=dim, grad=False, B=1, D=4 * rng.randrange(4, hi) if dim == 3 else 1,
                    H=4 * rng.randrange(4, hi), W=4 * rng.randrange(4, hi))
    return dict(kind=kind, dim=3, grad=True, B=rng.randrange(1, 5), D=4 * rng.randrange(4, 16),
                H=4 * rng.randrange(4, 16), W=4 * rng.randrange(4, 16))


# ---------------------------------------------------------------------------
# fields (torch, on the GPU).  Arrays are indexed [y, x] or [z, y, x]; level
# sets live on the half lattice, samples at lattice offsets (2i + off).
# ---------------------------------------------------------------------------
OFF = {2: dict(cell=(2, 2), node=(1, 1), u=(1, 2), v=(2, 1)),
       3: dict(cell=(2, 2, 2), u=(1, 2, 2), v=(2, 1, 2), w=(2, 2, 1), exy=(1, 1, 2), exz=(1, 2, 1), eyz=(2, 1, 1))}
FACES = {2: ("u", "v"), 3: ("u", "v", "w")}
SITES = {2: ("cell", "node"), 3: ("cell", "exy", "exz", "eyz")}


def _axes(xs):
    """Coordinates per axis (x first), shaped to broadcast over [z,] y, x."""
    d = len(xs)
    return [x.reshape([-1 if d - 1 - q == a else 1 for q in range(d)]) for a, x in enumerate(xs)]


def _at(kind, n, h):
    xs = []
    for d, o in enumerate(OFF[len(n)][kind]):
        m = n[d] + (o == 1)
        xs.append((2 * torch.arange(m, device="cuda", dtype=F64) + (o - 1)) * (h / 2))
    return _axes(xs)


def _lattice(n, h):
    return _axes([(torch.arange(2 * m + 3, device="cuda", dtype=F64) - 1) * (h / 2) for m in n])


def _shape(kind, n):
    return tuple(reversed([n[d] + (o == 1) for d, o in enumerate(OFF[len(n)][kind])]))


def _full(a, shape):
    return torch.as_tensor(a, dtype=F64, device="cuda").expand(shape).contiguous()


def _walls(X, ext):
    out = None
    for x, e in zip(X, ext):
        m = torch.minimum(x, e - x)
        out = m if out is None else torch.minimum(out, m)
    return out


def _r(X, c):
    return torch.sqrt(sum((x - float(q)) ** 2 for x, q in zip(X, c)))


class Fields:
    """The arrays of one problem: geometry from the case, u* (and a scale of
    the viscosity) from the seed."""

    def __init__(self, case, seed):
        kind = case["kind"]
        g = torch.Generator(device="cuda").manual_seed(int(seed))
        if kind == "jet2d":
            n = (case["n"], case["n"])
        else:
            n = tuple(case[k] for k in ("nx", "ny", "nz")[: 3 if case.get("dim", 3) == 3 and case.get("nz", 0) else 2])
        dim = len(n)
        self.n, self.dim = n, dim
        h = self.h = 1.0 / max(n)
        ext = [h * m for m in n]
        self.dt, self.floor = 0.01, FLOOR
        shape = case.get("shape", kind)
        rng = np.random.default_rng(case.get("geom", 0))
        L = _lattice(n, h)
        full = lambda a: _full(a, tuple(reversed([2 * m + 3 for m in n])))
        mu = lambda X: 1.0
        rho = lambda X: 1.0
        ubc = lambda d, X: 0.0
        noise = lambda d, shp: torch.rand(shp, generator=g, device="cuda", dtype=F64) * 2 - 1
        scale = 0.8 + 0.4 * float(torch.rand(1, generator=g, device="cuda", dtype=F64))
        solid = _walls(L, ext)
        if shape == "box":
            liquid = -1.0
        elif shape == "disk":
            liquid = _r(L, [e / 2 for e in ext]) - 0.3 * min(ext)
            mu = lambda X: scale
        elif shape == "bumps":
            # sum of eight Gaussians > 0.5, a moving solid disk (ball), log-uniform viscosity, two densities
            c = rng.uniform(0.2, 0.8, (8, dim)) * np.array(ext)
            s = rng.uniform(0.05, 0.12, 8) * min(ext)
            cs = rng.uniform(0.3, 0.7, dim) * np.array(ext)
            kk, th = rng.integers(1, 3, dim), rng.uniform(0.0, 1.0, dim)
            liquid = 0.5 - sum(torch.exp(-_r(L, c[i]) ** 2 / (2 * s[i] ** 2)) for i in range(8))
            ball = lambda X: _r(X, cs) - 0.1 * min(ext)
            solid = torch.minimum(solid, ball(L))

            def mu(X):
                m = torch.sin(2 * math.pi * (kk[0] * X[0] + th[0]))
                for d in range(1, dim):
                    m = m * torch.cos(2 * math.pi * (kk[d] * X[d] + th[d]))
                return scale * 10.0 ** (2.0 * m)
            rho = lambda X: torch.where(X[1] < 0.5 * ext[1], 1000.0, 1.0)
            ubc = lambda d, X: torch.where(ball(X) < _walls(X, ext), 0.5 if d == 0 else 0.0, 0.0)
        elif shape == "jet2d":
            # a wavy column of radius 0.03 falling onto a pool, inside a circle below a ceiling
            ph = float(rng.uniform(0, 2 * math.pi))
            x, y = L
            wave = 0.5 + 0.01 * torch.sin(20 * y + ph) * (0.8 - y)
            column = torch.maximum(torch.abs(x - wave) - 0.03, y - 0.8)
            pool = y - (0.2 + 0.01 * torch.cos(9 * x + ph))
            liquid = torch.minimum(column, pool)
            solid = torch.minimum(0.4 - _r(L, (0.5, 0.5)), 0.8 - y)
            self.source = full(torch.maximum(torch.abs(x - 0.5) - 0.03, 0.8 - y))
            self.dt = 0.002
            mu = lambda X: 0.075 * scale

            def ubc(d, X):
                ramp = torch.clamp((0.03 - torch.abs(X[0] - 0.5)) / h + 0.5, 0.0, 1.0)
                return -0.5 * ramp * (X[1] >= 0.8 - h / 4) if d else 0.0
            noise = lambda d, shp: _full(
                (-0.5 if d else 0.0) + 0.1 * scale * torch.sin(
                    6 * _at("uv"[d], n, h)[0] + 5 * _at("uv"[d], n, h)[1] + 7 * scale + d), shp)
        else:
            # liquid column of radius 0.05 about the vertical axis on a solid floor
            x, y, z = L
            r = torch.sqrt((x - 0.5 * ext[0]) ** 2 + (z - 0.5 * ext[2]) ** 2) - 0.05
            liquid = torch.maximum(r, y - 0.6 * ext[1])
            solid = torch.minimum(solid, y - 0.1 * ext[1])
            self.dt, self.floor = 1e-3, 0.0
            rho, mu = (lambda X: 1000.0), (lambda X: 10.0 * scale)
            noise = lambda d, shp: (-0.5 - 9.81e-3 if d == 1 else 0.0) + 0.05 * (
                torch.rand(shp, generator=g, device="cuda", dtype=F64) * 2 - 1)
        self.phi_liquid, self.phi_solid = full(liquid), full(solid)
        self.rho, self.ubc, self.ustar, self.mu = [], [], [], []
        for d, f in enumerate(FACES[dim]):
            X, shp = _at(f, n, h), _shape(f, n)
            self.rho.append(_full(rho(X), shp))
            self.ubc.append(_full(ubc(d, X), shp))
            self.ustar.append(noise(d, shp).contiguous())
        for s in SITES[dim]:
            self.mu.append(_full(mu(_at(s, n, h)), _shape(s, n)))

    def context(self):
        ctx = stokes.StokesContext(self.dim, self.n, self.h, self.dt)
        if self.floor:
            ctx.set_min_face_liquid(self.floor)
        return ctx

    def build(self, ctx):
        ctx.build_weights(self.phi_liquid, self.phi_solid, self.rho, self.mu, self.ubc)

    def outputs(self):
        n = self.n
        z = lambda k: torch.zeros(_shape(k, n), dtype=F64, device="cuda")
        u = [z(f) for f in FACES[self.dim]]
        tau = [z(k) for k in (("cell", "node") if self.dim == 2
                                                else ("cell", "cell", "exy", "exz", "eyz"))]
        return u, tau, z("cell")


def _vector(case, seed, ctx):
    """Random unknown vector in the context's slot layout (zero padding)."""
    lay, n = ctx.layout, ctx.n
    dt = F64 if case["precision"] == 0 else torch.float32
    x = torch.zeros(lay.total, dtype=dt, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    for f, v in enumerate(_field_views(x, lay, len(n))):
        k = _field_kind(f, len(n))
        w = v[tuple(slice(1, 1 + m) for m in _shape(k, n))]
        w.copy_(torch.randn(w.shape, generator=g, device="cuda", dtype=dt))
    return x


def _field_views(x, lay, dim):
    shp = (lay.rows, lay.pitch) if dim == 2 else (lay.planes, lay.rows, lay.pitch)
    size = int(np.prod(shp))
    return [x[f * lay.field_stride + lay.base:][:size].view(shp) for f in range(lay.nfields)]


def _field_kind(f, dim):
    return ("cell", "node", "cell")[f] if dim == 2 else ("cell", "cell", "exy", "exz", "eyz", "cell")[f]


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
class State:
    pass


def _net_layers(dim, cin, cout):
    return [(cin, 8, 3), (8, 8, 3), (8, 16, 3), (16, 16, 3), (16, 32, 3), (32, 32, 3), (48, 16, 3), (16, 16, 3),
            (24, 8, 3), (8, 8, 3), (8, cout, 1)]


def _net_problem(case, seed):
    """Per-layer weights [tap..., cin, cout] and biases, inputs and targets."""
    dim = case["dim"]
    cin, cout = (12, 8) if dim == 3 else (8, 4)
    nf = 6 if dim == 3 else 3
    rng = np.random.default_rng(seed)
    layers = []
    for ci, co, ks in _net_layers(dim, cin, cout):
        lim = math.sqrt(6.0 / (ci * ks ** dim))
        layers.append((rng.uniform(-lim, lim, (ks,) * dim + (ci, co)).astype(np.float32),
                       rng.uniform(-0.05, 0.05, co).astype(np.float32)))
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    shp = (case["B"], case["D"], case["H"], case["W"])
    x = torch.zeros(shp + (cin,), device="cuda")
    # Jacobi-scaled residual of unit RMS, then the logarithm of the inverse diagonal, as the solver feeds them
    x[..., :nf] = torch.randn(shp + (nf,), generator=g, device="cuda")
    x[..., nf:2 * nf] = torch.rand(shp + (nf,), generator=g, device="cuda") - 0.5
    y = torch.zeros(shp + (cout,), device="cuda")
    y[..., :nf] = torch.randn(shp + (nf,), generator=g, device="cuda")
    return cin, cout, layers, x, y


def _net_flat(layers):
    parts = []
    for w, b in layers:
        parts += [w.reshape(-1), b]
        parts.append(np.zeros(-sum(p.size for p in parts[-2:]) % 4, dtype=np.float32))
    return np.concatenate(parts)


def prepare(case, seed):
    s = State()
    s.case, kind = case, case["kind"]
    if kind == "net":
        cin, cout, layers, x, y = _net_problem(case, seed)
        s.shape = (case["B"], case["D"], case["H"], case["W"])
        s.net = stokes.Net(case["dim"], cin, cout, int(np.prod(s.shape)))
        s.net.set_params(_net_flat(layers))
        s.x, s.y = x, y
        return s
    if kind == "batch":
        s.fields, s.ctxs = [], []
        for i in range(case["count"]):
            rng = np.random.default_rng(case["geom"] + i)
            n = int(rng.integers(case["lo"], case["hi"] + 1))
            f = Fields(dict(kind="step2d", shape="bumps", nx=n, ny=n, dim=2, geom=case["geom"] + i), seed + 1000 * i)
            ctx = f.context()
            f.build(ctx)
            s.fields.append(f)
            s.ctxs.append(ctx)
        s.out = [f.outputs() for f in s.fields]
        s.batch = stokes.Batch(s.ctxs, stokes.default_options(mode=0, tol=1e-12, precond=case["precond"]))
        return s
    f = s.fields = Fields(case, seed)
    s.ctx = f.context()
    if kind == "apply":
        f.build(s.ctx)
        s.x = _vector(case, seed, s.ctx)
        s.y = torch.zeros_like(s.x)
        s.fields = None
        return s
    s.u, s.tau, s.p = f.outputs()
    if kind == "jet2d":
        s.u_star = [torch.empty_like(t) for t in f.ustar]
        s.phi = torch.empty_like(f.phi_liquid)
        s.opt = stokes.default_options(mode=stokes.FP32, precond=2, tol=1e-12)
        # the faces that carry u^n: all but fluid faces without liquid (export 2, bit 1)
        f.build(s.ctx)
        s.valid = ((s.ctx.export(2) & 2) == 0).to(torch.uint8)
    else:
        s.opt = stokes.default_options(mode=case["precision"], precond=case.get("precond", 0), tol=1e-12)
    return s


def run(s):
    kind = s.case["kind"]
    if kind == "apply":
        s.ctx.apply(s.x, s.y, s.case["precision"])
        return s.y
    if kind == "net":
        if s.case["grad"]:
            loss, grad = s.net.gradient(s.x, s.y, s.shape)
            return {"loss": loss, "grad": grad}
        return s.net.forward(s.x, s.shape)
    if kind == "batch":
        s.batch.solve([f.ustar for f in s.fields], [o[0] for o in s.out], [o[1] for o in s.out],
                      [o[2] for o in s.out])
        return [[*u, *tau, p] for u, tau, p in s.out]
    f = s.fields
    if kind == "jet2d":
        # u^n is the state's own velocity, so that every pass takes the same step
        s.ctx.advect(f.ustar, s.u_star, (0.0, -9.81), 8, phi_in=f.phi_liquid, phi_out=s.phi, valid=s.valid,
                     phi_union=f.source)
        s.ctx.build_weights(s.phi, f.phi_solid, f.rho, f.mu, f.ubc)
        s.ctx.solve_step(s.u_star, s.u, s.tau, s.p, s.opt)
        return {"u": s.u, "tau": s.tau, "p": s.p, "phi": s.phi}
    f.build(s.ctx)
    s.ctx.solve_step(f.ustar, s.u, s.tau, s.p, s.opt)
    return {"u": s.u, "tau": s.tau, "p": s.p}


def work(case):
    """Inputs read once and outputs written once; multiply-adds of one apply,
    or of the network's convolutions."""
    kind = case["kind"]
    if kind == "net":
        v = case["B"] * case["D"] * case["H"] * case["W"]
        dim = case["dim"]
        cin, cout = (12, 8) if dim == 3 else (8, 4)
        scale = [1, 1, 2 ** dim, 2 ** dim, 4 ** dim, 4 ** dim, 2 ** dim, 2 ** dim, 1, 1, 1]
        fl = sum(2.0 * v / q * ks ** dim * ci * co for q, (ci, co, ks) in zip(scale, _net_layers(dim, cin, cout)))
        return {"bytes": 4.0 * v * (cin + cout), "flops": fl * (3 if case["grad"] else 1)}
    if kind == "batch":
        m = (case["lo"] + case["hi"]) / 2
        slots, dim = case["count"] * m * m, 2
    else:
        n = (case["n"],) * 2 if kind == "jet2d" else [case[k] for k in ("nx", "ny", "nz") if case.get(k)]
        slots, dim = float(np.prod([m + 1 for m in n])), len(n)
    nf, nc = (3, 6) if dim == 2 else (6, 11)
    if kind == "apply":
        vec, coef = (8, 8) if case["precision"] == 0 else (4, 4 if case["precision"] == 1 else 2)
        return {"bytes": slots * (2 * nf * vec + nc * coef), "flops": slots * (40 if dim == 2 else 90)}
    faces, sites = dim, 2 if dim == 2 else 4
    return {"bytes": 8.0 * slots * (2 * 2 ** dim + 4 * faces + sites + nf), "flops": slots * (40 if dim == 2 else 90)}


# ---------------------------------------------------------------------------
# exact: the definition in 64 bits.  Every sample kind is held on the vertex
# lattice [z,] y, x; index i + 1 and i - 1 along an axis read zero outside.
# ---------------------------------------------------------------------------
def _simplex(v):
    """Fraction of a simplex (list of vertex values) where the linear interpolant is negative."""
    s = torch.sort(torch.stack(v, -1), -1).values
    a = [s[..., i] for i in range(len(v))]
    k = (s < 0).sum(-1)
    if len(v) == 3:
        one = a[0] * a[0] / ((a[0] - a[1]) * (a[0] - a[2]))
        rest = {2: 1.0 - a[2] * a[2] / ((a[2] - a[0]) * (a[2] - a[1]))}
    else:
        one = a[0] * a[0] * a[0] / ((a[0] - a[1]) * (a[0] - a[2]) * (a[0] - a[3]))
        x, y, p, q = a
        two = (x * x * y * y - (p + q) * x * y * (x + y) + p * q * (x * x + x * y + y * y)) / (
            (x - p) * (x - q) * (y - p) * (y - q))
        rest = {2: two, 3: 1.0 - q * q * q / ((q - x) * (q - y) * (q - p))}
    out = torch.where(k == len(v), 1.0, 0.0).to(F64)
    out = torch.where(k == 1, one, out)
    for m, e in rest.items():
        out = torch.where(k == m, e, out)
    return out


def _fraction(phi, off, n):
    """Fraction of {phi < 0} of every control volume of a kind, on the vertex lattice (0 where none exists)."""
    dim = len(n)
    V = tuple(reversed([m + 1 for m in n]))
    m = [n[d] + (off[d] == 1) for d in range(dim)]

    def at(o):
        return phi[tuple(slice(off[d] + o[d], off[d] + o[d] + 2 * m[d] - 1, 2) for d in reversed(range(dim)))]
    cube = [(i, j) if dim == 2 else (i, j, k) for k in ((-1, 0, 1) if dim == 3 else (0,)) for j in (-1, 0, 1)
            for i in (-1, 0, 1)]
    neg = pos = False
    for o in cube:
        neg, pos = neg | (at(o) < 0), pos | (at(o) > 0)
    f = (neg & ~pos).to(F64)
    mix = neg & pos
    val = {o: at(o)[mix] for o in cube}
    if dim == 2:
        ring = [(1, 0), (1, 1), (0, 1), (-1, 1), (-1, 0), (-1, -1), (0, -1), (1, -1)]
        tot = sum(_simplex([val[0, 0], val[ring[t]], val[ring[(t + 1) % 8]]]) for t in range(8)) / 8.0
    else:
        tot = 0.0
        for axis in range(3):
            for sg in (-1, 1):
                c = [0, 0, 0]
                c[axis] = sg
                ua, va = [d for d in range(3) if d != axis]
                cor = []
                for a, b in ((-1, -1), (1, -1), (1, 1), (-1, 1)):
                    o = list(c)
                    o[ua], o[va] = a, b
                    cor.append(tuple(o))
                for t in range(4):
                    tot = tot + _simplex([val[0, 0, 0], val[tuple(c)], val[cor[t]], val[cor[(t + 1) % 4]]])
        tot = tot / 24.0
    f[mix] = tot
    out = torch.zeros(V, dtype=F64, device="cuda")
    out[tuple(slice(0, k) for k in f.shape)] = f
    return out


class Exact:
    """Weights and the operator A = C + B K B^T in 64 bits."""

    def __init__(self, F, phi_liquid=None):
        dim, n = F.dim, F.n
        self.dim, self.n = dim, n
        self.V = tuple(reversed([m + 1 for m in n]))
        phi = F.phi_liquid if phi_liquid is None else phi_liquid
        WL = {k: _fraction(phi, o, n) for k, o in OFF[dim].items()}
        WF = {}
        for k, o in OFF[dim].items():
            WF[k] = self.lift((1.0 - _fraction(F.phi_solid, o, n))[self.real(k)], k)
        self.pair = {(0, 1): "node"} if dim == 2 else {(0, 1): "exy", (0, 2): "exz", (1, 2): "eyz"}
        stress = [self.edge(0, 1)] if dim == 2 else list(self.pair.values())
        zero = {k: (WL[k] > 0) & (WF[k] == 0) for k in ["cell"] + stress}
        self.K, self.rec, self.wf, self.live, bad = [], [], [], [], []
        for d, f in enumerate(FACES[dim]):
            wf, wl = WF[f].clone(), WL[f]
            ax = dim - 1 - d
            wf.select(ax, 0).zero_()
            wf.select(ax, n[d]).zero_()
            inval = zero["cell"] | self.sh(zero["cell"], d, -1)
            for e in range(dim):
                if e != d:
                    z = zero[self.edge(d, e)]
                    inval = inval | z | self.sh(z, e, 1)
            wf = torch.where(inval, torch.zeros_like(wf), wf)
            live = (wf > 0) & (wl > 0)
            mass = self.lift(F.rho[d], f) * torch.clamp(wl, min=F.floor)
            nul = torch.zeros_like(wf)
            self.K.append(torch.where(live, F.dt * wf / mass, nul))
            self.rec.append(torch.where(live, F.dt / mass, nul))
            self.wf.append(wf)
            self.live.append(live)
            bad.append((wf > 0) & ~(wl > 0))
        self.ubc = [self.lift(F.ubc[d], f) for d, f in enumerate(FACES[dim])]
        any2 = lambda m, d, s: m[d] | self.sh(m[d], d if s is None else s, 1 if s is None else -1)
        b = l = False
        for d in range(dim):
            b, l = b | any2(bad, d, None), l | any2(self.live, d, None)
        inv_h = 1.0 / F.h
        act = (WL["cell"] > 0) & ~b & l
        nul = torch.zeros(self.V, dtype=F64, device="cuda")
        one = torch.ones_like(nul)
        muc = self.lift(F.mu[0], "cell")
        self.a = {"cell": torch.where(act, WL["cell"] * inv_h, nul)}
        self.d = {"cell": torch.where(act, WL["cell"] * WF["cell"] / muc, one)}
        self.act, self.WF = {"cell": act}, WF
        for q, ((d, e), k) in enumerate(self.pair.items()):
            b = any2(bad, d, e) | any2(bad, e, d)
            l = any2(self.live, d, e) | any2(self.live, e, d)
            act = (WL[k] > 0) & ~b & ((WF[k] > 0) | l)
            self.a[k] = torch.where(act, WL[k] * inv_h, nul)
            self.d[k] = torch.where(act, WL[k] * WF[k] / self.lift(F.mu[1 + q], k), one)
            self.act[k] = act

    def edge(self, d, e):
        return self.pair[(min(d, e), max(d, e))]

    def real(self, kind):
        return tuple(slice(0, m) for m in _shape(kind, self.n))

    def lift(self, a, kind):
        out = torch.zeros(self.V, dtype=F64, device="cuda")
        out[self.real(kind)] = a.reshape(_shape(kind, self.n))
        return out

    def sh(self, a, d, s):
        """a at index + s along axis d (x = 0), zero outside."""
        ax = self.dim - 1 - d
        out = torch.zeros_like(a)
        m = a.shape[ax]
        if s > 0:
            out.narrow(ax, 0, m - 1).copy_(a.narrow(ax, 1, m - 1))
        else:
            out.narrow(ax, 1, m - 1).copy_(a.narrow(ax, 0, m - 1))
        return out

    def stresses(self):
        return ["node"] if self.dim == 2 else ["exy", "exz", "eyz"]

    def bt(self, x):
        """B^T x on every face; x: unknown fields in slot order."""
        a = self.a["cell"]
        p = x[-1]
        if self.dim == 2:
            c, s = [a * (p - x[0]), a * (p + x[0])], {"node": self.a["node"] * x[1]}
        else:
            c = [a * (p - x[0]), a * (p - x[1]), a * (p + x[0] + x[1])]
            s = {k: self.a[k] * x[2 + i] for i, k in enumerate(self.stresses())}
        out = []
        for d in range(self.dim):
            z = c[d] - self.sh(c[d], d, -1)
            for e in range(self.dim):
                if e != d:
                    t = s[self.edge(d, e)]
                    z = z + (t - self.sh(t, e, 1))
            out.append(z)
        return out

    def b_of(self, z):
        """Rows of D and G^T applied to face values z (without the row weights)."""
        g = [self.sh(z[d], d, 1) - z[d] for d in range(self.dim)]     # u_x, v_y(, w_z)
        p = -sum(g)
        cells = [g[0] - g[1]] if self.dim == 2 else [g[0] - g[2], g[1] - g[2]]
        edges = []
        for (d, e) in self.pair:
            edges.append((z[d] - self.sh(z[d], e, -1)) + (z[e] - self.sh(z[e], d, -1)))
        return cells + edges + [p]

    def kinds(self):
        return [_field_kind(f, self.dim) for f in range(3 if self.dim == 2 else 6)]

    def apply(self, x):
        z = [k * t for k, t in zip(self.K, self.bt(x))]
        rows = self.b_of(z)
        out = []
        for f, k in enumerate(self.kinds()):
            y = self.a[k] * rows[f]
            if f < len(x) - 1:
                if k == "cell" and self.dim == 3:
                    y = y + torch.where(self.act["cell"], self.d[k] * (x[f] + 0.5 * x[1 - f]), x[f])
                else:
                    y = y + self.d[k] * x[f]
            else:
                y = torch.where(self.act["cell"], y, x[f])
            out.append(y)
        return out

    def rhs(self, ustar):
        us = [self.lift(u, f) for u, f in zip(ustar, FACES[self.dim])]
        v = [w * u + (1.0 - w) * b for w, u, b in zip(self.wf, us, self.ubc)]
        rv, rb = self.b_of(v), self.b_of(self.ubc)
        return [self.a[k] * (rv[f] - (1.0 - self.WF[k]) * rb[f]) for f, k in enumerate(self.kinds())]

    def diagonal(self):
        near = lambda d: self.K[d] + self.sh(self.K[d], d, 1)
        s = [near(d) for d in range(self.dim)]
        a2 = self.a["cell"] ** 2
        dc = self.d["cell"]
        if self.dim == 2:
            cells, p = [dc + a2 * (s[0] + s[1])], a2 * (s[0] + s[1])
        else:
            cells, p = [dc + a2 * (s[0] + s[2]), dc + a2 * (s[1] + s[2])], a2 * (s[0] + s[1] + s[2])
        edges = []
        for (d, e), k in self.pair.items():
            t = self.K[d] + self.sh(self.K[d], e, -1) + self.K[e] + self.sh(self.K[e], d, -1)
            edges.append(self.d[k] + self.a[k] ** 2 * t)
        act = self.act["cell"]
        one = torch.ones_like(p)
        return [torch.where(act, c, one) for c in cells] + edges + [torch.where(act, p, one)]

    def solve(self, b, seconds=12.0):
        """Jacobi-PCG to a recurrence residual of 1e-14 (None if it takes too long)."""
        import time
        began = time.monotonic()
        b = torch.stack(b)
        minv = 1.0 / torch.stack(self.diagonal())
        x, r = torch.zeros_like(b), b.clone()
        z = minv * r
        p, rz, stop = z.clone(), (r * z).sum(), 1e-28 * float((b * b).sum())
        for it in range(200000):
            q = torch.stack(self.apply(list(p)))
            al = rz / (p * q).sum()
            x += al * p
            r -= al * q
            z = minv * r
            new = (r * z).sum()
            p = z + (new / rz) * p
            rz = new
            if it % 16 == 15:
                if float((r * r).sum()) <= stop:
                    return list(x)
                if time.monotonic() - began > seconds:
                    return None
        return None

    def step(self, ustar):
        x = self.solve(self.rhs(ustar))
        if x is None:
            return None
        u = []
        for d, (f, t) in enumerate(zip(FACES[self.dim], self.bt(x))):
            us = self.lift(ustar[d], f)
            v = torch.where(self.live[d], us - self.rec[d] * t, torch.where(self.wf[d] == 0, self.ubc[d], us))
            u.append(v[self.real(f)].contiguous())
        fields = [torch.where(self.act[k], v, torch.zeros_like(v))[self.real(k)].contiguous()
                  for v, k in zip(x, self.kinds())]
        return {"u": u, "tau": fields[:-1], "p": fields[-1]}


def _exact_net(case, seed):
    dim = case["dim"]
    cin, cout, layers, x, y = _net_problem(case, seed)
    conv = torch.nn.functional.conv2d if dim == 2 else torch.nn.functional.conv3d
    pool = torch.nn.functional.avg_pool2d if dim == 2 else torch.nn.functional.avg_pool3d
    up = lambda t: torch.nn.functional.interpolate(t, scale_factor=2, mode="nearest")
    perm = (dim + 1, dim) + tuple(range(dim))
    P = [(torch.from_numpy(w).cuda().to(F64).permute(perm).contiguous(), torch.from_numpy(b).cuda().to(F64))
         for w, b in layers]
    first = lambda t: t.permute(0, 4, 1, 2, 3).to(F64) if dim == 3 else t[:, 0].permute(0, 3, 1, 2).to(F64)

    def cv(i, t):
        w, b = P[i]
        t = conv(t, w, b, padding=w.shape[-1] // 2)
        return torch.relu(t) if i < 10 else t
    with torch.no_grad():
        e0 = cv(1, cv(0, first(x)))
        e1 = cv(3, cv(2, pool(e0, 2)))
        e2 = cv(5, cv(4, pool(e1, 2)))
        d1 = cv(7, cv(6, torch.cat([up(e2), e1], 1)))
        out = cv(10, cv(9, cv(8, torch.cat([up(d1), e0], 1))))
    if case["grad"]:
        t = first(y)
        loss = (((out - t) ** 2).flatten(1).sum(1) / (t ** 2).flatten(1).sum(1)).mean()
        return {"loss": float(loss), "grad": None}
    return out.movedim(1, -1).reshape(-1).contiguous()


def exact(case, seed):
    kind = case["kind"]
    if kind == "net":
        return _exact_net(case, seed)
    if kind == "batch" or (kind == "step2d" and case["shape"] == "bumps"):
        return None                      # tens of thousands of plain iterations
    F = Fields(case, seed)
    if kind == "apply":
        E = Exact(F)
        ctx = F.context()                # for its layout of vectors alone
        lay, n = ctx.layout, F.n
        x = _vector(case, seed, ctx)
        ctx.close()
        cut = [tuple(slice(1, 1 + m) for m in E.V) for _ in E.kinds()]
        xs = [v[c].to(F64) for v, c in zip(_field_views(x, lay, F.dim), cut)]
        y = torch.zeros(lay.total, dtype=F64, device="cuda")
        for v, c, k, t in zip(_field_views(y, lay, F.dim), cut, E.kinds(), E.apply(xs)):
            v[c] = t
        return y
    if kind == "jet2d":
        return None                      # its transport has kinks (clamped bilinear interpolation)
    return Exact(F).step(F.ustar)
