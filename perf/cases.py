"""Measured cases: the calls that programs of this library make, through its
public binding (`paper_1602_05806_gb300.sdg`, `.autograd`), over the range of
grids, degrees, precisions and options the library is used with.

    listed()             the named cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  inputs on the device and the handle a program keeps
    run(state)           one pass through the public entry points
    work(case)           bytes and operations a pass cannot do without
    exact(case, seed)    what run() returns, evaluated in 64 bits with torch
                         alone (systems solved in Fourier space), on the same
                         inputs

Grid sizes, degrees and time steps are those of `workloads.py` (8x8 N=3,
64x64 N=5, 256x256 N=7, 48^3 N=4, the batch of uneven members) and generic
ones around them.  Every initial state is a Taylor-Green vortex plus a
divergence-free perturbation of random Fourier modes drawn from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1602_05806_gb300 import autograd as sdg_autograd
from paper_1602_05806_gb300 import sdg

TWO_PI = 2.0 * math.pi
THETA = 0.51
# as tight as the small solves of the tests: the solver raises it to three
# times the residual that rounding the solution to FP64 leaves
RTOL = 1e-13


# ------------------------------------------------------------------ the cases
def _case(name, kind, n, N, nu, dt, nsub=1, precision="mixed", **more):
    n = tuple(n)
    c = dict(kind=kind, dim=len(n), nx=n[0], ny=n[1], nz=n[2] if len(n) == 3 else 1, N=N, nu=nu, dt=dt,
             nsub=nsub, precision=precision)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    big = dict(n=(256, 256), N=7, nu=1e-3, dt=2e-3, nsub=5)
    mid = dict(n=(64, 64), N=5, nu=0.01, dt=5e-3, nsub=3)
    cube = dict(n=(48, 48, 48), N=4, nu=1.0 / 1600, dt=1e-3)
    return [
        # the operator alone, as a program with its own Krylov solver or
        # preconditioner calls it: FP32 in 2D, FP64 in 3D
        _case("apply_2d_256_N7_f32", "apply", precision="f32", op="pressure", **big),
        _case("apply_3d_48_N4_f64", "apply", precision="f64", op="viscous", **cube),
        # explicit convection alone (operator splitting around the caller's
        # own implicit part), five sub-steps
        _case("convect_2d_256_N7", "convect", **big),
        # the non-iterative stages of a caller-driven step: projections to the
        # main grid and back, pressure right-hand side, velocity update
        _case("stages_3d_48_N4", "stages", **cube),
        # the two linear solves alone: few iterations on a large 3D grid, a
        # plain FP64 solve of an ordinary size, the longest mixed solve
        _case("viscous_cg_3d_48_N4", "viscous_cg", **cube),
        _case("pressure_cg_2d_64_N5_f64", "pressure_cg", **dict(mid, precision="f64")),
        _case("pressure_cg_2d_256_N7", "pressure_cg", **big),
        # whole time steps: the smallest run (FP64, the default precision),
        # an ordinary 2D one, the 3D one
        _case("step_2d_8_N3_f64", "step", n=(8, 8), N=3, nu=0.1, dt=0.01, precision="f64"),
        _case("step_2d_64_N5", "step", **mid),
        _case("step_3d_48_N4", "step", **cube),
        # gradient of a loss through one step (forward and backward)
        _case("gradient_2d_32_N5", "gradient", **dict(mid, n=(32, 32))),
        # uneven independent problems stepped together
        _case("batch_2d_12", "batch", n=(64, 64), N=7, nu=1e-3, dt=1e-3,
              members="64x4 16x7 32x3 16x2 32x6 64x3 16x4 32x7 16x5 64x2 32x4 16x6"),
    ]


# relative cost of one pass, for keeping drawn cases within the listed ones:
# iterations of a solve grow with cells per side times (N + 1)^2, and small
# grids pay for launches
def _cost(c):
    n1 = c["N"] + 1
    ndof = c["nx"] * c["ny"] * c["nz"] * n1 ** c["dim"]
    one = ndof + 2e5
    its = max(c["nx"], c["ny"], c["nz"]) * n1 * n1
    f64 = 15.0 if c["precision"] == "f64" else 1.0
    if c["kind"] in ("apply", "convect", "stages"):
        return one * 10 * c["nsub"]
    if c["kind"] == "viscous_cg":
        return one * 200 * f64
    return one * its * f64 * {"pressure_cg": 1.0, "step": 1.3, "gradient": 3.0, "batch": 1.0}[c["kind"]]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


# degree of a 2D solve: odd degrees on moderate grids only (on larger ones
# FP64 itself fixes their pressure to about 1e-9: the near-kernel modes)
def _degree(rng, cells):
    return rng.choice([2, 3, 4, 5, 6, 7] if cells <= 40 else [2, 4, 6])


def draw(rng):
    limit = _cost(dict(_case("", "pressure_cg", (256, 256), 7, 0, 0)))
    while True:
        kind = rng.choice(["apply", "apply", "convect", "stages", "viscous_cg", "pressure_cg", "pressure_cg", "step",
                           "step", "gradient", "batch"])
        if kind == "batch":
            k = rng.randint(4, 14)
            members = " ".join("%dx%d" % (m, _degree(rng, m)) for m in (int(_log(rng, 8, 64)) for _ in range(k)))
            return _case("", kind, (64, 64), 7, _log(rng, 1e-4, 1e-1), 1e-3, members=members,
                         precision=rng.choice(["mixed", "mixed", "mixed", "f64"]) if k < 7 else "mixed")
        dim = rng.choice([2, 2, 3])
        free = kind in ("apply", "convect", "stages")
        if dim == 2:
            a = _log(rng, 6, 256)
            n = (max(4, int(a)), max(4, min(256, int(a * _log(rng, 0.5, 2)))))
            N = rng.randint(1, 11) if free else _degree(rng, max(n))
        else:
            N = rng.randint(1, 6) if free else rng.randint(1, 4)
            a = _log(rng, 4, 48)
            n = tuple(max(3, min(48, int(a * _log(rng, 0.6, 1.6)))) for _ in range(3))
        nsub = rng.choice([1, 1, 2, 3, 5])
        # CFL about 0.4 per sub-step for velocities of order one
        dt = nsub * 0.4 / ((2 * N + 1) * sum(n) / TWO_PI)
        more = {}
        if kind == "apply":
            precision = rng.choice(["f32", "f64"])
            more["op"] = rng.choice(["pressure", "viscous"])
        elif kind in ("convect", "stages"):
            precision = "mixed"
        else:
            precision = rng.choice(["mixed", "mixed", "f64"])
        c = _case("", kind, n, N, _log(rng, 1e-4, 1e-1), min(dt, 0.01), nsub=nsub, precision=precision, **more)
        ndof = math.prod(n) * (N + 1) ** dim
        if _cost(c) <= (0.3 if kind not in ("apply", "convect", "stages") else 1.0) * limit and ndof <= 48 ** 3 * 5 ** 3:
            return c


# ------------------------------------------------------------------ inputs
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _grid(c):
    return (c["nx"], c["ny"], c["nz"])[:c["dim"]]


def _state(c, seed, ref):
    """Velocity on the dual grids and pressure: Taylor-Green plus ten random
    divergence-free modes (wave numbers up to 6, amplitude about 0.02)."""
    rng = np.random.default_rng(seed)
    dim = c["dim"]
    modes = [(rng.integers(-6, 7, dim), rng.uniform(0, TWO_PI), rng.normal(size=3) * 0.01) for _ in range(10)]
    U = []
    for d in range(dim):
        x = ref.coords(d)
        if dim == 2:
            u = torch.sin(x[0]) * torch.cos(x[1]) if d == 0 else -torch.cos(x[0]) * torch.sin(x[1])
        else:
            u = (torch.sin(x[0]) * torch.cos(x[1]) * torch.cos(x[2]) if d == 0 else
                 -torch.cos(x[0]) * torch.sin(x[1]) * torch.cos(x[2]) if d == 1 else torch.zeros(ref.shape, **ref.kw))
        u = u.clone()
        for k, phase, a in modes:
            k = [float(v) for v in k] + [0.0] * (3 - dim)
            m = max(1.0, max(abs(v) for v in k))
            # curl of a plane-wave vector potential (2D: of a e_z)
            amp = (k[1] * a[2], -k[0] * a[2]) if dim == 2 else (
                k[1] * a[2] - k[2] * a[1], k[2] * a[0] - k[0] * a[2], k[0] * a[1] - k[1] * a[0])
            u = u + (amp[d] / m) * torch.cos(sum(k[e] * x[e] for e in range(dim)) + phase)
        U.append(u.expand(ref.shape).contiguous())
    x = ref.coords(None)
    if dim == 2:
        P = 0.25 * (torch.cos(2 * x[0]) + torch.cos(2 * x[1]))
    else:
        P = (torch.cos(2 * x[0]) + torch.cos(2 * x[1])) * (torch.cos(2 * x[2]) + 2.0) / 16.0
    return U, P.expand(ref.shape).contiguous()


def _member_cases(c):
    out = []
    for i, m in enumerate(c["members"].split()):
        cells, N = (int(v) for v in m.split("x"))
        nu = c["nu"] * (1.0 + 0.5 * (i % 3))
        out.append(_case("", "step", (cells, cells), N, nu, c["dt"], precision=c["precision"]))
    return out


def _inputs(c, seed):
    """(reference, dict of tensors): everything run() is given besides the handle."""
    ref = _Ref(c)
    U, P = _state(c, seed, ref)
    kind = c["kind"]
    if kind == "apply":
        # a Krylov vector: smooth part and noise of every scale
        g = torch.Generator(device=P.device).manual_seed(int(seed))
        x = P + U[0] + 0.1 * torch.randn(ref.shape, generator=g, **ref.kw)
        return ref, {"x": x.float() if c["precision"] == "f32" else x}
    if kind == "convect":
        return ref, {"V": [ref.dual_to_main(U[d], d).contiguous() for d in range(ref.dim)]}
    if kind == "viscous_cg":
        F = ref.rk3([ref.dual_to_main(U[d], d) for d in range(ref.dim)])[0]
        return ref, {"b": ref.mass_all(F).contiguous(), "x0": F.contiguous()}
    if kind == "pressure_cg":
        b = ref.rhs(ref.ustar(U), P)
        return ref, {"b": (b - ref.kernel_part(b)).contiguous(), "x0": P}
    if kind == "stages":
        # Pn: the pressure a caller's own solver returned
        return ref, {"U": U, "P": P, "Pn": P + 0.01 * U[0]}
    if kind == "gradient":
        W, _ = _state(c, seed + 1, ref)
        vol = math.prod(ref.dx)
        # cotangents of a quadratic misfit against another state
        lamU = [(vol * ref.mass_all(U[d] - 0.9 * W[d])).contiguous() for d in range(ref.dim)]
        return ref, {"U": U, "P": P, "lamU": lamU, "lamP": (0.1 * vol * ref.mass_all(P - 0.5 * U[0])).contiguous()}
    return ref, {"U": U, "P": P}


def _handle(c, h=None):
    if h is None:
        dim = c["dim"]
        h = sdg.Handle(dim, _grid(c), (TWO_PI,) * dim, c["N"], c["nu"], THETA, c["dt"])
    h.set_options(sdg.SDG_FP64 if c["precision"] == "f64" else sdg.SDG_MIXED, RTOL, RTOL)
    h.set_convection_substeps(c["nsub"])
    return h


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "batch":
        members = _member_cases(c)
        b = sdg.Batch([(m["dim"], _grid(m), (TWO_PI,) * m["dim"], m["N"], m["nu"]) for m in members], THETA, c["dt"])
        data = []
        for i, m in enumerate(members):
            _handle(m, b.members[i])
            data.append(_inputs(m, seed * 1000 + i)[1])
        return {"kind": "batch", "batch": b, "data": data}
    ref, data = _inputs(c, seed)
    like = data["U"][0] if "U" in data else data["V"][0] if "V" in data else data.get("x", data.get("b"))
    s = dict(kind=c["kind"], h=_handle(c), op=c.get("op"), **data)
    s["new"] = lambda: torch.empty_like(like)
    if c["kind"] == "gradient":
        s["nu"] = torch.tensor(c["nu"], dtype=torch.float64)
    return s


# ------------------------------------------------------------------ one pass
def run(state):
    s, kind = state, state["kind"]
    if kind == "batch":
        for h, d in zip(s["batch"].members, s["data"]):
            h.set_state(d["U"], d["P"])
        s["batch"].step(1)
        out = []
        for h, d in zip(s["batch"].members, s["data"]):
            U, P = [torch.empty_like(d["P"]) for _ in range(h.dim)], torch.empty_like(d["P"])
            h.get_state(U, P)
            out.append({"U": U, "P": P})
        return out
    h, new = s["h"], s["new"]
    if kind == "apply":
        y = new()
        (h.pressure_apply if s["op"] == "pressure" else h.viscous_apply)(s["x"], y)
        return y
    if kind == "convect":
        F = [new() for _ in range(h.dim)]
        h.convect(s["V"], F)
        return F
    if kind == "stages":
        V = [new() for _ in range(h.dim)]
        W = [new() for _ in range(h.dim)]
        for d in range(h.dim):
            h.dual_to_main(d, s["U"][d], V[d])
            h.main_to_dual(d, V[d], W[d])
        b = new()
        h.pressure_rhs(W, s["P"], b)
        Un = [new() for _ in range(h.dim)]
        h.velocity_update(W, s["Pn"], s["P"], Un)
        return {"V": V, "W": W, "b": b, "U": Un}
    if kind in ("viscous_cg", "pressure_cg"):
        x = s["x0"].clone()
        (h.viscous_cg if kind == "viscous_cg" else h.pressure_cg)(s["b"], x)
        return x
    if kind == "step":
        h.set_state(s["U"], s["P"])
        h.step(1)
        U, P = [new() for _ in range(h.dim)], new()
        h.get_state(U, P)
        return {"U": U, "P": P}
    # gradient
    U0 = [u.clone().requires_grad_(True) for u in s["U"]]
    P0 = s["P"].clone().requires_grad_(True)
    nu = s["nu"].clone().requires_grad_(True)
    U, P = sdg_autograd.steps(h, U0, P0, nu, 1)
    g = torch.autograd.grad([*U, P], [*U0, P0, nu], [*s["lamU"], s["lamP"]])
    return {"U": [u.detach() for u in U], "P": P.detach(), "dU": list(g[:-2]), "dP": g[-2], "dnu": g[-1]}


# ------------------------------------------------------------------ work
# pressure iterations on these states (they set the operations a solve cannot
# do without): in proportion to cells (N + 1)^2, more for odd degrees; a
# viscous solve takes about fifteen
def _iterations(c):
    n1 = c["N"] + 1
    per = 1.0 if c["dim"] == 3 else 1.5 if c["N"] % 2 else 0.5
    return per * max(_grid(c)) * n1 * n1


def work(case):
    c = dict(case)
    if c["kind"] == "batch":
        parts = [work(m) for m in _member_cases(c)]
        return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}
    n1, dim = c["N"] + 1, c["dim"]
    ndof = math.prod(_grid(c)) * n1 ** dim
    size = 4 if c["precision"] == "f32" else 8
    apply_flops = ndof * dim * (3 * n1 + 4)      # three n1 x n1 blocks per line, halved by their mirror symmetry
    project = ndof * 4 * n1
    convect = ndof * dim * dim * (2 * n1 + 12) * 3 * c["nsub"]
    rhs = apply_flops + ndof * dim * 4 * n1
    update = ndof * dim * 4 * n1
    its = _iterations(c)
    iteration = apply_flops + 10 * ndof
    vis = 15 * iteration
    kind = c["kind"]
    if kind == "apply":
        return {"bytes": 2 * ndof * size, "flops": apply_flops}
    if kind == "convect":
        return {"bytes": 2 * dim * ndof * 8, "flops": convect}
    if kind == "stages":
        return {"bytes": (4 * dim + 2) * ndof * 8, "flops": 2 * dim * project + rhs + update}
    if kind == "viscous_cg":
        return {"bytes": 3 * ndof * 8, "flops": vis}
    if kind == "pressure_cg":
        return {"bytes": 3 * ndof * 8, "flops": its * iteration}
    step = 2 * dim * project + convect + dim * vis + rhs + its * iteration + update
    if kind == "step":
        return {"bytes": 2 * (dim + 1) * ndof * 8, "flops": step}
    return {"bytes": 5 * (dim + 1) * ndof * 8, "flops": 3 * step}


# ------------------------------------------------------------------ 64-bit reference
def exact(case, seed):
    c = dict(case)
    with torch.no_grad():
        if c["kind"] == "batch":
            return [dict(zip(("U", "P"), r.step(d["U"], d["P"])))
                    for r, d in (_inputs(m, seed * 1000 + i) for i, m in enumerate(_member_cases(c)))]
        ref, s = _inputs(c, seed)
        kind, dims = c["kind"], range(c["dim"])
        if kind == "apply":
            x = s["x"].double()
            return ref.theta * ref.aprime(x) if c["op"] == "pressure" else ref.mass_all(x) + ref.nu * ref.aprime(x)
        if kind == "convect":
            return ref.rk3(s["V"])
        if kind == "stages":
            V = [ref.dual_to_main(s["U"][d], d) for d in dims]
            W = [ref.main_to_dual(V[d], d) for d in dims]
            b = ref.rhs(W, s["P"])
            return {"V": V, "W": W, "b": b, "U": ref.velocity(W, ref.theta * s["Pn"] + (1 - ref.theta) * s["P"])}
        if kind == "viscous_cg":
            return ref.solve(s["b"], 1.0, ref.nu)
        if kind == "pressure_cg":
            x = ref.solve(s["b"], 0.0, ref.theta)
            return x - ref.kernel_part(x) + ref.kernel_part(s["x0"])
        if kind == "step":
            return dict(zip(("U", "P"), ref.step(s["U"], s["P"])))
    U0 = [u.clone().requires_grad_(True) for u in s["U"]]
    P0 = s["P"].clone().requires_grad_(True)
    nu = torch.tensor(c["nu"], **ref.kw).requires_grad_(True)
    ref.nu = nu
    U, P = ref.step(U0, P0)
    g = torch.autograd.grad([*U, P], [*U0, P0, nu], [*s["lamU"], s["lamP"]])
    return {"U": [u.detach() for u in U], "P": P.detach(), "dU": list(g[:-2]), "dP": g[-2], "dnu": g[-1].cpu()}


class _Solve(torch.autograd.Function):
    """x = (cmass M + scale A')^-1 b; backward by the symmetry of the system."""

    @staticmethod
    def forward(ctx, ref, b, cmass, scale):
        x = ref.refined(b, cmass, float(scale))
        ctx.ref, ctx.cmass, ctx.scale = ref, cmass, float(scale)
        ctx.save_for_backward(x)
        return x

    @staticmethod
    def backward(ctx, g):
        mu = ctx.ref.refined(g, ctx.cmass, ctx.scale)
        ds = -(mu * ctx.ref.aprime(ctx.saved_tensors[0])).sum() if ctx.needs_input_grad[3] else None
        return None, mu, None, ds


class _Ref:
    """The semi-implicit staggered DG step of a periodic box in FP64 torch:
    1D matrices by quadrature of their defining integrals, whole-array
    contractions, exact solves in Fourier space."""

    def __init__(self, c):
        self.dim, self.n, self.N = c["dim"], _grid(c), c["N"]
        self.n1 = n1 = self.N + 1
        self.nu, self.theta, self.dt, self.nsub = c["nu"], THETA, c["dt"], c["nsub"]
        self.dx = [TWO_PI / v for v in self.n]
        self.kw = dict(dtype=torch.float64, device=_device())
        self.shape = tuple(reversed(self.n)) + (n1,) * self.dim
        x, w = np.polynomial.legendre.leggauss(n1)
        self.xi, w = 0.5 * (x + 1), 0.5 * w
        s, q = np.polynomial.legendre.leggauss(n1 + 3)
        s, q = 0.5 * (s + 1), 0.5 * q
        lo, hi = self.phi(0.5 * s), self.phi(0.5 + 0.5 * s)          # (n1, points)
        dlo, dhi = self.dphi(0.5 * s), self.dphi(0.5 + 0.5 * s)
        p0, p1, ph = (self.phi(np.array([v]))[:, 0] for v in (0.0, 1.0, 0.5))
        ip = lambda a, b: (a * q) @ b.T  # noqa: E731
        Rt = np.outer(ph, p0) + 0.5 * ip(hi, dlo)
        Lt = np.outer(ph, p1) - 0.5 * ip(lo, dhi)
        Rb = np.outer(p1, ph) - 0.5 * ip(dhi, lo)
        Lb = np.outer(p0, ph) + 0.5 * ip(dlo, hi)
        wi = np.diag(1.0 / w)
        HR, HL, HC = -Rb @ wi @ Rt, -Lb @ wi @ Lt, Rb @ wi @ Lt + Lb @ wi @ Rt
        Dn = self.dphi(self.xi).T                                     # Dn[k, m] = phi_m'(xi_k)
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), **self.kw)  # noqa: E731
        self.w, self.p0, self.p1 = t(w), t(p0), t(p1)
        self.Rt, self.Lt, self.Rb, self.Lb = t(Rt), t(Lt), t(Rb), t(Lb)
        self.wRt, self.wLt = t(wi @ Rt), t(wi @ Lt)
        self.ML, self.MR = t(wi @ (0.5 * ip(lo, hi))), t(wi @ (0.5 * ip(hi, lo)))
        self.HR, self.HL, self.HC = t(HR), t(HL), t(HC)
        self.DW = t(wi @ Dn.T @ np.diag(w))
        self.wp0, self.wp1 = t(wi @ p0), t(wi @ p1)
        # local patterns whose repetition in every cell has no weak gradient
        _, sv, vt = np.linalg.svd(Rt - Lt)
        null = vt[sv <= 1e-10 * max(1.0, np.abs(Rt).max())]
        self.K1 = t(null.T @ null)
        self.np = dict(HR=HR, HL=HL, HC=HC, w=w)
        self.sym = None

    # Lagrange basis through the Gauss-Legendre nodes and its derivative
    def phi(self, x):
        return np.array([np.prod([(x - b) / (a - b) for b in self.xi if b != a], axis=0) * np.ones_like(x)
                         for a in self.xi])

    def dphi(self, x):
        out = np.zeros((self.n1, len(x)))
        for i, a in enumerate(self.xi):
            for m, c in enumerate(self.xi):
                if m != i:
                    out[i] += np.prod([(x - b) / (a - b) for j, b in enumerate(self.xi) if j not in (i, m)],
                                      axis=0) * np.ones_like(x) / (a - c)
        return out

    def eax(self, d):
        return self.dim - 1 - d

    def lax(self, d):
        return 2 * self.dim - 1 - d

    def on(self, v, d, ax):
        shp = [1] * (2 * self.dim)
        shp[ax(d)] = -1
        return v.reshape(shp)

    def coords(self, dual):
        out = []
        for d in range(self.dim):
            i = np.arange(self.n[d])[:, None] + (0.5 if dual == d else 0.0) + self.xi[None, :]
            shp = [1] * (2 * self.dim)
            shp[self.eax(d)], shp[self.lax(d)] = self.n[d], self.n1
            out.append(torch.as_tensor(i * self.dx[d], **self.kw).reshape(shp))
        return out

    def along(self, Z, X, d):
        return torch.movedim(torch.movedim(X, self.lax(d), -1) @ Z.T, -1, self.lax(d))

    def shift(self, X, d, s):
        return torch.roll(X, s, self.eax(d))

    def mass_perp(self, X, d):
        for e in range(self.dim):
            if e != d:
                X = X * self.on(self.w, e, self.lax)
        return X

    def mass_all(self, X):
        return self.mass_perp(X, -1)

    def aprime(self, X):
        out = 0.0
        for d in range(self.dim):
            H = (self.along(self.HL, self.shift(X, d, 1), d) + self.along(self.HC, X, d)
                 + self.along(self.HR, self.shift(X, d, -1), d))
            out = out + (self.dt / self.dx[d] ** 2) * self.mass_perp(H, d)
        return out

    def dual_to_main(self, U, d):
        return self.along(self.ML, self.shift(U, d, 1), d) + self.along(self.MR, U, d)

    def main_to_dual(self, F, d):
        return self.along(self.ML, F, d) + self.along(self.MR, self.shift(F, d, -1), d)

    def face(self, X, d, v):
        return torch.movedim(X, self.lax(d), -1) @ v

    def convection(self, V):
        out = [0.0] * self.dim
        for d in range(self.dim):
            ax, minus = self.eax(d), [self.face(V[c], d, self.p1) for c in range(self.dim)]
            plus = [torch.roll(self.face(V[c], d, self.p0), -1, ax) for c in range(self.dim)]
            s = 2.0 * torch.maximum(minus[d].abs(), plus[d].abs())
            for c in range(self.dim):
                f = 0.5 * (minus[c] * minus[d] + plus[c] * plus[d]) - 0.5 * s * (plus[c] - minus[c])
                surf = f[..., None] * self.wp1 - torch.roll(f, 1, ax)[..., None] * self.wp0
                vol = self.along(self.DW, V[c] * V[d], d)
                out[c] = out[c] - (torch.movedim(surf, -1, self.lax(d)) - vol) / self.dx[d]
        return out

    def rk3(self, V):
        k = self.dt / self.nsub
        for _ in range(self.nsub):
            V1 = [v + k * a for v, a in zip(V, self.convection(V))]
            V2 = [0.75 * v + 0.25 * (u + k * a) for v, u, a in zip(V, V1, self.convection(V1))]
            V = [v / 3.0 + (2.0 / 3.0) * (u + k * a) for v, u, a in zip(V, V2, self.convection(V2))]
        return V

    def rhs(self, Us, P):
        out = -(1.0 - self.theta) * self.aprime(P)
        for d in range(self.dim):
            D = self.along(self.Rb, Us[d], d) - self.along(self.Lb, self.shift(Us[d], d, 1), d)
            out = out - self.mass_perp(D, d) / self.dx[d]
        return out - out.mean()

    def velocity(self, Us, q):
        return [Us[d] - (self.dt / self.dx[d]) * (self.along(self.wRt, self.shift(q, d, -1), d)
                                                  - self.along(self.wLt, q, d)) for d in range(self.dim)]

    def kernel_part(self, X):
        m = X.mean(dim=tuple(range(self.dim)), keepdim=True)
        for d in range(self.dim):
            m = self.along(self.K1, m, d)
        return m.expand(self.shape)

    # block-circulant solves: Fourier over the elements, eigenvectors of the 1D symbols over the nodes
    def symbols(self):
        if self.sym is None:
            self.sym, ws = [], 1.0 / np.sqrt(self.np["w"])
            for d in range(self.dim):
                z = np.exp(1j * TWO_PI * np.arange(self.n[d]) / self.n[d])[:, None, None]
                S = self.np["HL"] / z + self.np["HC"] + self.np["HR"] * z
                S = 0.5 * (S + S.conj().transpose(0, 2, 1))
                lam, vec = np.linalg.eigh(ws[:, None] * S * ws[None, :])
                self.sym.append((torch.as_tensor(lam, **self.kw), torch.as_tensor(vec, device=self.kw["device"])))
        return self.sym

    def per_wave(self, X, M, d):
        X = torch.movedim(X, (self.eax(d), self.lax(d)), (0, -1))
        Y = (X.reshape(X.shape[0], -1, self.n1) @ M.transpose(1, 2)).reshape(X.shape)
        return torch.movedim(Y, (0, -1), (self.eax(d), self.lax(d)))

    def spectral(self, b, cmass, scale):
        ax = tuple(range(self.dim))
        half = [self.on(self.w.sqrt(), d, self.lax) for d in ax]
        Y = torch.fft.fftn(b, dim=ax)
        den = torch.full((1,) * (2 * self.dim), cmass, **self.kw)
        for d in ax:
            lam, vec = self.symbols()[d]
            Y = self.per_wave(Y / half[d], vec.conj().transpose(1, 2), d)
            shp = [1] * (2 * self.dim)
            shp[self.eax(d)], shp[self.lax(d)] = lam.shape
            den = den + scale * self.dt / self.dx[d] ** 2 * lam.reshape(shp)
        ok = den.abs() > 1e-11 * den.abs().max()
        Y = torch.where(ok, Y / torch.where(ok, den, torch.ones_like(den)), torch.zeros_like(Y))
        for d in ax:
            Y = self.per_wave(Y, self.symbols()[d][1], d) / half[d]
        return torch.fft.ifftn(Y, dim=ax).real.contiguous()

    def refined(self, b, cmass, scale):
        op = lambda v: cmass * self.mass_all(v) + scale * self.aprime(v)  # noqa: E731
        x = self.spectral(b, cmass, scale)
        for _ in range(2):
            x = x + self.spectral(b - op(x), cmass, scale)
        return x

    def solve(self, b, cmass, scale):
        return _Solve.apply(self, b, cmass, scale)

    def ustar(self, U):
        F = self.rk3([self.dual_to_main(U[d], d) for d in range(self.dim)])
        return [self.main_to_dual(self.solve(self.mass_all(F[d]), 1.0, self.nu), d) for d in range(self.dim)]

    def step(self, U, P):
        Us = self.ustar(U)
        x = self.solve(self.rhs(Us, P), 0.0, self.theta)
        x = x - self.kernel_part(x) + self.kernel_part(P)
        Pn = x - self.mass_all(x).sum() / math.prod(self.n)
        return self.velocity(Us, self.theta * Pn + (1.0 - self.theta) * P), Pn
