"""Performance cases of the CNP discontinuous Galerkin framework.

Each case is work that a program using the framework has it do, through the
Python binding's public methods: applications of the operator (R, J v, J^T w)
in its three arithmetics, the residual as a differentiable function, the
set-up and application of the preconditioner, and whole Newton solves. The
meshes are boxes with the boundary conditions of the repository's workloads
(unit-cube and plate-reactor electrolytes, a three-ion channel, the
manufactured-solution square), at sizes from a handful of elements to the full
workloads.

``exact`` evaluates the same quantities with dense 64-bit tensor arithmetic
(torch einsum over explicit basis matrices, torch's own differentiation),
without the framework's kernels.
"""
import functools
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2112_09271_gb300 as enp

WALL, INLET, OUTLET, DIRICHLET, ELECTRODE0 = 1, 2, 3, 4, 5

# ------------------------------------------------------------------ the cases


def listed():
    return [
        # The manufactured-solution square: the smallest problem users run (convergence
        # studies, unit tests). One residual and one J v, where launches are everything.
        dict(name="quads_8x8_p2", kind="quads", nx=8, ny=8, p=2),
        # A small plate reactor carrying eight operating points: J v in double-float
        # arithmetic as the outer Krylov operator of a voltage sweep. Latency-bound.
        dict(name="jvp_df_reactor_24x6x2_p2_b8", kind="jvp_df", family="reactor", nx=24, ny=6, nz=2,
             p=2, batch=8),
        # The default arithmetic (native FP64) on the mid-size cube: residual, J v and
        # J^T w, as an adjoint-based optimisation calls them.
        dict(name="ops_f64_cube_16x16x16_p3", kind="ops_f64", family="cube", nx=16, ny=16, nz=16,
             p=3, batch=1),
        # The headline operator: J v at FP64 accuracy on the three-ion channel.
        dict(name="jvp_df_channel_64x32x16_p3", kind="jvp_df", family="channel", nx=64, ny=32, nz=16,
             p=3, batch=1),
        # The differentiable residual: forward, and backward to the state and to the
        # physical parameters (inverse design, parameter fitting).
        dict(name="grad_df_cube_24x24x24_p2", kind="grad_df", family="cube", nx=24, ny=24, nz=24,
             p=2, batch=1),
        # The inner operator of the mixed-precision solver at full size.
        dict(name="jvp_f32_channel_64x32x16_p3", kind="jvp_f32", family="channel", nx=64, ny=32,
             nz=16, p=3, batch=1),
        # The same at the highest degree, on an odd mesh with graded spacing and two points.
        dict(name="jvp_f32_reactor_61x15x5_p4_b2", kind="jvp_f32", family="reactor", nx=61, ny=15,
             nz=5, p=4, batch=2),
        # Preconditioner refresh of a Newton step and its first application, three
        # fields at p = 3 (192 unknowns per element), full size.
        dict(name="setup_f32_channel_64x32x16_p3", kind="setup_f32", family="channel", nx=64, ny=32,
             nz=16, p=3, batch=1),
        # The same at p = 4 with two fields (250 unknowns per element).
        dict(name="setup_f32_reactor_48x12x4_p4", kind="setup_f32", family="reactor", nx=48, ny=12,
             nz=4, p=4, batch=1),
        # One application of the preconditioner a long channel gets by default (downwind
        # sweep, plus the coarse potential correction), inside FP32 Krylov iterations.
        dict(name="precond_f32_reactor_192x48x16_p2", kind="precond_f32", family="reactor", nx=192,
             ny=48, nz=16, p=2, batch=1),
        # A whole mixed-precision Newton solve of the three-ion channel to 1e-10.
        dict(name="newton_channel_40x20x10_p3", kind="newton", family="channel", nx=40, ny=20, nz=10,
             p=3, batch=1),
        # A whole solve of eight operating points of a small reactor as one batch, the
        # Newton iterations driven on the device.
        dict(name="newton_reactor_24x6x2_p2_b8", kind="newton", family="reactor", nx=24, ny=6, nz=2,
             p=2, batch=8),
    ]


# per kind: (fewest, most) unknowns per element times elements times points, and degrees
_RANGE = {
    "quads": (2e2, 2e5, (1, 2, 3)),
    "jvp_df": (1e4, 6e6, (1, 2, 3, 4)),
    "ops_f64": (1e4, 6e5, (1, 2, 3, 4)),
    "grad_df": (1e4, 7e5, (1, 2, 3)),
    "jvp_f32": (1e4, 8e6, (1, 2, 3, 4)),
    "setup_f32": (1e4, 5e5, (1, 2, 3, 4)),
    "precond_f32": (2e4, 3e6, (1, 2, 3)),
    "newton": (1e4, 6e5, (1, 2, 3)),
}


def draw(rng):
    kind = rng.choice(list(_RANGE))
    lo, hi, degrees = _RANGE[kind]
    p = rng.choice(degrees)
    dof = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    if kind == "quads":
        cells = max(4.0, dof / (2 * (p + 1) ** 2))
        nx = max(2, round(math.sqrt(cells) * math.exp(rng.uniform(-0.5, 0.5))))
        return dict(kind=kind, nx=nx, ny=max(2, round(cells / nx)), p=p)
    family = rng.choice(("cube", "channel", "reactor"))
    batch = rng.choice((1, 1, 1, 2, 3, 8)) if kind != "setup_f32" else 1
    m = 3 if family == "channel" else 2
    cells = max(12.0, dof / (m * (p + 1) ** 3 * batch))
    shape = {"cube": (1, 1, 1), "channel": (4, 2, 1), "reactor": (12, 3, 1)}[family]
    s = (cells / (shape[0] * shape[1] * shape[2])) ** (1 / 3)
    n = [max(lo_, round(c * s * math.exp(rng.uniform(-0.25, 0.25)))) for c, lo_ in zip(shape, (3, 2, 1))]
    if kind == "precond_f32" and rng.random() < 0.4:  # a long channel: the downwind sweep
        family, m = "reactor", 2
        n = [rng.randint(128, 192), max(2, round(math.sqrt(cells / 160 * 3))), 1]
        n[2] = max(1, round(cells / (n[0] * n[1])))
    while n[0] * n[1] * n[2] * m * (p + 1) ** 3 * batch > hi and max(n) > 3 and kind != "precond_f32":
        n[n.index(max(n))] -= 1
    if kind == "newton":
        family = "reactor" if batch > 1 else family
    return dict(kind=kind, family=family, nx=n[0], ny=n[1], nz=n[2], p=p, batch=batch)


# ------------------------------------------------------------- the problems


def _problem(case, seed):
    """Mesh, boundary tags and physical parameters; the operating conditions
    (inlet concentrations, diffusivities, potentials) vary with the seed."""
    r = np.random.RandomState(seed % (2 ** 31) ^ 0x5EED)
    vary = lambda x: float(x * (1 + 0.05 * r.uniform(-1, 1)))  # noqa: E731
    p = case["p"]
    if case["kind"] == "quads":
        n, length, dim, family = [case["nx"], case["ny"]], [1.0, 1.0], 2, "quads"
    else:
        n, dim, family = [case["nx"], case["ny"], case["nz"]], 3, case["family"]
        length = {"cube": [1.0, 1.0, 1.0], "channel": [4.0, 2.0, 1.0], "reactor": [12.0, 3.0, 1.0]}[family]
    coords = [np.linspace(0.0, L, k + 1) for L, k in zip(length, n)]
    if case["kind"] == "jvp_f32" and family == "reactor":  # graded towards the electrodes
        t = coords[1] / length[1]
        coords[1] = length[1] * (t - 0.5 / (2 * math.pi) * np.sin(2 * math.pi * t))
    tags = []
    for s in range(2 * dim):
        others = [b for b in range(dim) if b != s // 2]
        t = np.full([n[b] for b in reversed(others)], DIRICHLET if dim == 2 else WALL, dtype=np.uint8)
        if dim == 3 and s < 2:
            t[:] = INLET if s == 0 else OUTLET
        if dim == 3 and s in (2, 3):
            x = 0.5 * (coords[0][1:] + coords[0][:-1])
            lo, hi = (5.0, 7.0) if family == "reactor" else (length[0] / 3, 2 * length[0] / 3)
            t[:, (x > lo) & (x < hi)] = ELECTRODE0 + (s - 2)
        tags.append(t.reshape(-1))
    P = SimpleNamespace(dim=dim, n_el=n + [1] * (3 - dim), coords=coords, tags=tags, p=p, q=p + 2,
                        F=1.0, RT=1.0, C_IP=10.0, bv_oxidant=-1, bv_J0=0.0, bv_alpha1=0.5,
                        bv_alpha2=0.5, bv_n=1.0, bv_gamma=1.0, bv_c_ref=1.0, bv_phi_app=[0.0] * 4,
                        bv_J0_axis=-1, bv_J0_lo=0.0, bv_J0_hi=1.0, vel_kind=1)
    if family == "quads":
        P.m, P.z, P.D, P.c_in = 2, [1.0, -1.0], [vary(1e-3), vary(2e-3)], [1.0, 1.0]
        P.vel_kind, P.vel_params = 0, [1.0, 0.5, 0.0]
    elif family == "cube":
        P.m, P.z, P.D, P.c_in = 2, [1.0, -1.0], [vary(1e-3), vary(2e-3)], [vary(1.0), 1.0]
        P.vel_params = [0, 1, 0.0, 1.0, 1.0]
        P.bv_oxidant, P.bv_J0, P.bv_phi_app = 0, 0.1, [vary(1.17), 0.0, 0.0, 0.0]
    elif family == "channel":
        P.m, P.z = 3, [1.0, -1.0, 2.0]
        P.D, P.c_in = [vary(5e-4), vary(1e-3), vary(2e-3)], [vary(1.0), vary(2.0), 0.5]
        P.vel_params = [0, 1, 0.0, 2.0, 5.0]
        P.bv_oxidant, P.bv_J0, P.bv_n, P.bv_c_ref = 2, 0.1, 2.0, 0.5
        P.bv_phi_app = [vary(1.17), 0.0, 0.0, 0.0]
    else:
        P.m, P.z, P.D, P.c_in = 2, [2.0, -2.0], [vary(1e-4), vary(1.48e-4)], [vary(1.0), 1.0]
        P.vel_params = [0, 1, 0.0, 3.0, 1.0]
        P.bv_oxidant, P.bv_J0, P.bv_n = 0, 0.05, 2.0
        P.bv_phi_app = [vary(0.03 * 38.92), 0.0, 0.0, 0.0]
        P.bv_J0_axis = 2
    P.E, P.Np, P.NBF = int(np.prod(n)), (p + 1) ** dim, int(sum(len(t) for t in tags))
    batch = case.get("batch", 1)
    # applied potentials of the operating points, 0.01 to 0.05 V
    P.phi = None
    if batch > 1:
        P.phi = np.zeros((batch, 4))
        P.phi[:, 0] = 38.92 * np.linspace(0.01, 0.05, batch) * (1 + 0.05 * r.uniform(-1, 1, batch))
    return P


def _inputs(P, case, seed):
    """A state near the inlet composition and directions in [-1, 1]."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    batch = case.get("batch", 1)
    shape = (batch, P.m, P.E, P.Np)
    rnd = lambda *s: torch.rand(s, generator=g, device="cuda", dtype=torch.float64) * 2 - 1  # noqa: E731
    u = rnd(*shape)
    u[:, 0] *= 0.1
    for k in range(1, P.m):
        u[:, k] = P.c_in[k - 1] * (1 + 0.1 * u[:, k])
    return u.reshape(-1), rnd(*shape).reshape(-1), rnd(*shape).reshape(-1), rnd


def prepare(case, seed):
    P = _problem(case, seed)
    kind, batch = case["kind"], case.get("batch", 1)
    u, v, w, rnd = _inputs(P, case, seed)
    op = enp.Operator(P, batch=batch)
    if P.phi is not None:
        op.set_phi_app(P.phi)
    S = SimpleNamespace(kind=kind, op=op, u=u, v=v, w=w, out=[torch.empty_like(u) for _ in range(3)])
    if kind.endswith("_df") or kind in ("newton", "grad_df"):
        op.set_arithmetic(enp.ARITH_DF32)
    if kind == "quads":
        S.src, S.dir = _boundary_data(P, rnd)
        op.set_sources(S.src.reshape(-1), S.dir.reshape(-1))
    if kind.endswith("_f32"):
        S.u32, S.v32, S.out32 = u.float(), v.float(), torch.empty_like(u, dtype=torch.float32)
    if kind == "grad_df":
        S.fn = enp.residual_function(op)
        S.u = u.requires_grad_(True)
        S.theta = torch.zeros(op.n_theta, dtype=torch.float64, device="cuda", requires_grad=True)
    if kind == "precond_f32":
        op.set_preconditioner(1)
        op.block_jacobi_setup(u, enp.BJ_F32)
    if kind == "newton":
        op.set_preconditioner(1)
        S.u = torch.empty_like(u).reshape(batch, P.m, -1)
        S.u[:, 0] = 0.0 if batch == 1 else torch.tensor(0.5 * P.phi[:, :1], device="cuda")
        for k in range(1, P.m):
            S.u[:, k] = P.c_in[k - 1]
        S.u = S.u.reshape(-1)
    return S


def run(S):
    op = S.op
    if S.kind == "quads":
        return op.residual(S.u, out=S.out[0]), op.jvp(S.u, S.v, out=S.out[1])
    if S.kind == "jvp_df":
        return op.jvp(S.u, S.v, out=S.out[0])
    if S.kind == "ops_f64":
        return (op.residual(S.u, out=S.out[0]), op.jvp(S.u, S.v, out=S.out[1]),
                op.vjp(S.u, S.w, out=S.out[2]))
    if S.kind == "jvp_f32":
        return op.jvp_f32(S.u32, S.v32, out=S.out32)
    if S.kind == "grad_df":
        S.u.grad = S.theta.grad = None
        r = S.fn(S.u, S.theta)
        r.backward(S.w)
        return r.detach(), S.u.grad, S.theta.grad
    if S.kind == "setup_f32":
        op.block_jacobi_setup(S.u, enp.BJ_F32)
        return op.block_jacobi_apply_f32(S.v32, out=S.out32)
    if S.kind == "precond_f32":
        return op.block_jacobi_apply_f32(S.v32, out=S.out32)
    u = S.u.clone()
    op.newton_solve(u, max_it=30, rtol=1e-10, krylov_restart=50, krylov_max_it=4000, krylov_rtol=1e-3,
                    mixed=True, bj_storage=enp.BJ_BF16 if op.batch == 1 else enp.BJ_F32,
                    device_loop=op.batch > 1)
    return u


def work(case):
    """Inputs read once, outputs written once; floating-point operations of the
    sum-factorised contractions (and of inversion and products for blocks)."""
    P = _problem(case, 0)
    kind, batch, m, p, dim = case["kind"], case.get("batch", 1), P.m, P.p, P.dim
    n, q = p + 1, p + 2
    nb, dof = m * P.Np, m * P.Np * P.E * batch
    if dim == 3:
        vol = n * n * q * n + n * q * q * n + q ** 3 * n + 3 * q ** 4
        face = 2 * (n * n * n + 2 * (n * n * q + n * q * q)) / 2  # value and derivative, per side
        el = lambda nv: 2 * m * ((nv + 1) * vol + 6 * (nv + 1) * face)  # noqa: E731
    else:
        vol = n * q * n + q * q * n + 2 * q ** 3
        el = lambda nv: 2 * m * ((nv + 1) * vol + 4 * (nv + 1) * 3 * n * q)  # noqa: E731
    app = lambda nv: el(nv) * P.E * batch  # noqa: E731
    if kind == "quads":
        return {"bytes": 8.0 * (3 * dof + 2 * dof), "flops": app(1) + app(2)}
    if kind == "jvp_df":
        return {"bytes": 24.0 * dof, "flops": app(2)}
    if kind == "ops_f64":
        return {"bytes": 8.0 * (2 + 3 + 3) * dof, "flops": app(1) + 2 * app(2)}
    if kind == "jvp_f32":
        return {"bytes": 12.0 * dof, "flops": app(2)}
    if kind == "grad_df":
        return {"bytes": 8.0 * (2 + 3) * dof, "flops": app(1) + app(2)}
    if kind == "setup_f32":  # the stored inverses are an output
        return {"bytes": P.E * 4.0 * nb * nb + 16.0 * dof, "flops": 2.0 * P.E * nb ** 3}
    if kind == "precond_f32":
        return {"bytes": P.E * batch * 4.0 * nb * nb + 8.0 * dof, "flops": 2.0 * P.E * batch * nb * nb}
    # a solve: Newton steps of about 100 inner iterations, each one preconditioner
    # application (16-bit or 32-bit inverses) and one FP32 J v
    its = 400
    return {"bytes": its * (P.E * batch * (2.0 if batch == 1 else 4.0) * nb * nb + 20.0 * dof),
            "flops": its * app(2)}


# ------------------------------------------- the same quantities in 64 bits


def _boundary_data(P, rnd):
    src = rnd(P.m, P.E, P.q ** P.dim)
    dirv = 0.1 * rnd(P.m, P.NBF, P.q ** (P.dim - 1))
    dirv[1:] += 1.0
    return src, dirv


@functools.lru_cache(None)
def _tables(p):
    """Gauss points and weights, Lagrange basis on the Gauss-Lobatto nodes: values
    and derivatives at the Gauss points, derivatives at the two ends."""
    L = np.polynomial.legendre
    xg, wg = L.leggauss(p + 2)
    inner = L.Legendre.basis(p).deriv().roots() if p > 1 else np.array([])
    nodes = np.concatenate([[-1.0], np.sort(inner.real), [1.0]])
    V = np.linalg.inv(np.polynomial.polynomial.polyvander(nodes, p))  # columns: basis coefficients
    at = lambda x, c: np.polynomial.polynomial.polyval(x, c).T  # noqa: E731
    dV = np.polynomial.polynomial.polyder(V)
    dev = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda", dtype=torch.float64)  # noqa: E731
    return dev(xg), dev(wg), dev(at(xg, V)), dev(at(xg, dV)), dev(at(np.array([-1.0, 1.0]), dV))


class _Dense:
    """The discretisation with plain tensor operations. A state is a tensor
    [batch, field, (ez,) ey, ex, (nz,) ny, nx]: the element and node axes of
    direction a are at position -1 - a - dim and -1 - a."""

    def __init__(self, P, batch, src=None, dirv=None):
        self.P, self.batch, self.dim = P, batch, P.dim
        self.xg, self.wg, self.B, self.dB, self.dL = _tables(P.p)
        self.src, self.dirv = src, dirv
        d = P.dim
        self.grid = list(reversed(P.n_el[:d]))
        self.shape = [batch, P.m] + self.grid + [P.p + 1] * d
        self.xv = [torch.tensor(c, device="cuda") for c in P.coords]
        self.h = [x[1:] - x[:-1] for x in self.xv]
        self.theta = dict(D=torch.tensor(P.D, device="cuda", dtype=torch.float64),
                          cin=torch.tensor(P.c_in, device="cuda", dtype=torch.float64),
                          phi=(torch.tensor(P.bv_phi_app, device="cuda", dtype=torch.float64)
                               .expand(batch, 4) if P.phi is None
                               else torch.tensor(P.phi, device="cuda")))

    def el(self, x, a):
        """Per-element values along axis a, broadcast over a point array."""
        return x.reshape([-1] + [1] * (a + self.dim))

    def along(self, M, t, a):
        return torch.movedim(torch.tensordot(t, M, dims=([t.dim() - 1 - a], [1])), -1, t.dim() - 1 - a)

    def back(self, M, t, a):
        return self.along(M.T, t, a)

    def split(self, u):
        """Library layout [batch, field, element, node] -> the tensor."""
        return u.reshape(self.shape)

    def coefs(self):
        P, t = self.P, self.theta
        z, D = P.z, t["D"]
        mu = D / P.RT
        mig = [z[k] * mu[k] * P.F for k in range(P.m)]
        a = [P.F * z[k] * (D[k] - D[-1]) for k in range(P.m - 1)]
        kap = [z[k] * (z[k] * mu[k] - z[-1] * mu[-1]) * P.F ** 2 for k in range(P.m - 1)]
        return D, mig, a, kap

    def points(self, a, shape_dim):
        """Coordinates along axis a at the Gauss points, broadcastable."""
        x = self.xv[a][:-1, None] + 0.5 * (self.xg + 1) * self.h[a][:, None]
        return x.reshape([x.shape[0]] + [1] * (shape_dim - 1) + [x.shape[1]] + [1] * a)

    def velocity(self, x):
        """The velocity components from the coordinates (a list of tensors)."""
        P, v = self.P, self.P.vel_params
        if P.vel_kind == 0:
            return [v[a] for a in range(self.dim)]
        s = x[int(v[1])] - v[2]
        ua = 6 * v[4] / v[3] ** 2 * s * (v[3] - s)
        return [ua if a == int(v[0]) else 0.0 for a in range(self.dim)]

    def volume(self, U):
        P, d = self.P, self.dim
        D, mig, ak, kc = self.coefs()
        full, grads = U, []
        for a in range(d):
            g = U
            for b in range(d):
                g = self.along(self.dB if a == b else self.B, g, b)
            grads.append(g * self.el(2 / self.h[a], a))
        for b in range(d):
            full = self.along(self.B, full, b)
        vel = self.velocity([self.points(a, d) for a in range(d)])
        w = 1.0
        for a in range(d):
            w = w * self.wg.reshape([-1] + [1] * a) * self.el(0.5 * self.h[a], a)
        kappa = sum(kc[k] * full[:, k + 1] for k in range(P.m - 1))
        G = []
        for a in range(d):
            g = grads[a]
            rows = [kappa * g[:, 0] + sum(ak[k] * g[:, k + 1] for k in range(P.m - 1))]
            for k in range(P.m - 1):
                rows.append(D[k] * g[:, k + 1] - full[:, k + 1] * (vel[a] - mig[k] * g[:, 0]))
            G.append(torch.stack(rows, 1))
        out = 0.0
        for a in range(d):
            t = w * G[a] * self.el(2 / self.h[a], a)
            for b in range(d):
                t = self.back(self.dB if a == b else self.B, t, b)
            out = out + t
        if self.src is not None:
            q = P.q
            t = -w * self.src.reshape([1, P.m] + self.grid + [q] * d)
            for b in range(d):
                t = self.back(self.B, t, b)
            out = out + t
        return out

    def trace(self, U, a, end):
        """(value, outward-agnostic reference derivative along +a) at the face
        points of each element's end 0 or 1 of axis a."""
        pos = U.dim() - 1 - a
        val = U.select(pos, -1 if end else 0).unsqueeze(pos)
        der = self.along(self.dL[end:end + 1], U, a)
        for b in range(self.dim):
            if b != a:
                val, der = self.along(self.B, val, b), self.along(self.B, der, b)
        return val, der

    def lift(self, S, T, a, end):
        """Rows of an element from the value and reference-derivative coefficients."""
        for b in range(self.dim):
            if b != a:
                S, T = self.back(self.B, S, b), self.back(self.B, T, b)
        unit = torch.zeros(self.P.p + 1, 1, device="cuda", dtype=torch.float64)
        unit[-1 if end else 0] = 1
        return self.along(unit, S, a) + self.along(self.dL[end:end + 1].T, T, a)

    def cross(self, a):
        """Face weights and coordinates off axis a."""
        w, x = 1.0, [None] * self.dim
        for b in range(self.dim):
            if b != a:
                w = w * self.wg.reshape([-1] + [1] * b) * self.el(0.5 * self.h[b], b)
                x[b] = self.points(b, self.dim)
        return w, x

    def diagonal(self, a, ha):
        s = self.el(ha ** 2, a)
        for b in range(self.dim):
            if b != a:
                s = s + self.el(self.h[b] ** 2, b)
        return torch.sqrt(s)

    def interior(self, a, lo, hi, hl, hu):
        """Rows of the lower and upper elements from the faces between them; lo and
        hi: states of the elements below and above, hl and hu their sizes along a."""
        P = self.P
        D, mig, ak, kc = self.coefs()
        cm, dm = self.trace(lo, a, 1)
        cp, dp = self.trace(hi, a, 0)
        scl, scu = self.el(2 / hl, a), self.el(2 / hu, a)
        dm, dp = dm * scl, dp * scu
        w, x = self.cross(a)
        x[a] = torch.zeros(1, device="cuda", dtype=torch.float64)  # the plate flow varies off its axis only
        un = self.velocity(x)[a]
        delta = P.C_IP * P.p ** 2 / (0.5 * (self.diagonal(a, hl) + self.diagonal(a, hu)))
        S, T, TP = [None], [None], [None]
        km = sum(kc[k] * cm[:, k + 1] for k in range(P.m - 1))
        kp = sum(kc[k] * cp[:, k + 1] for k in range(P.m - 1))
        jphi = cm[:, 0] - cp[:, 0]
        T0 = S0 = 0.0
        for k in range(P.m - 1):
            f = k + 1
            jc = cm[:, f] - cp[:, f]
            qm, qp = un - mig[k] * dm[:, 0], un - mig[k] * dp[:, 0]
            S.append(-0.5 * D[k] * (dm[:, f] + dp[:, f]) + D[k] * delta * jc
                     + 0.5 * (cm[:, f] * qm + cp[:, f] * qp) + 0.25 * torch.abs(qm + qp) * jc)
            T.append(-0.5 * D[k] * jc)
            TP.append(0.5 * D[k] * jc)
            T0 = T0 - 0.5 * ak[k] * jc
            S0 = S0 - 0.5 * ak[k] * (dm[:, f] + dp[:, f])
        T[0], TP[0] = T0 - 0.5 * km * jphi, -(T0 - 0.5 * kp * jphi)
        S[0] = S0 - 0.5 * (km * dm[:, 0] + kp * dp[:, 0]) + 0.5 * delta * (km + kp) * jphi
        S, T, TP = (torch.stack(t, 1) * w for t in (S, T, TP))
        return self.lift(S, scl * T, a, 1), self.lift(-S, -scu * TP, a, 0)

    def boundary(self, a, end, U):
        P = self.P
        D, mig, ak, kc = self.coefs()
        nrm = 1.0 if end else -1.0
        ha = self.h[a][-1:] if end else self.h[a][:1]
        sc = 2 / ha.item() * nrm
        c, d = self.trace(U, a, end)
        d = d * sc
        w, x = self.cross(a)
        x[a] = self.xv[a][-1 if end else 0]
        vel = self.velocity(x)[a]
        un = vel * nrm
        others = [self.grid[i] if i != self.dim - 1 - a else 1 for i in range(self.dim)]
        tag = torch.tensor(P.tags[2 * a + end].astype(np.int64), device="cuda").reshape(others + [1] * self.dim)
        zero = torch.zeros_like(c[:, 0])
        S, T = [zero] * P.m, [zero] * P.m
        for k in range(P.m - 1):
            S[k + 1] = torch.where(tag == INLET, un * self.theta["cin"][k] + zero, S[k + 1])
            S[k + 1] = torch.where(tag == OUTLET, (un - mig[k] * d[:, 0]) * c[:, k + 1], S[k + 1])
        if P.bv_oxidant >= 0:
            ox = P.bv_oxidant
            co = (c[:, ox + 1] if ox < P.m - 1
                  else -sum(P.z[k] * c[:, k + 1] for k in range(P.m - 1)) / P.z[-1])
            J0 = P.bv_J0
            if P.bv_J0_axis >= 0:
                half = 0.5 * (P.bv_J0_hi - P.bv_J0_lo)
                r = (x[P.bv_J0_axis] - P.bv_J0_lo - half) / half
                J0 = 0.6 * J0 * (2 - r * r)
            f = P.bv_n * P.F / P.RT
            for j in range(2):
                phi = self.theta["phi"][:, j].reshape([self.batch] + [1] * (2 * self.dim))
                on = tag == ELECTRODE0 + j
                eta = torch.where(on, phi - c[:, 0], zero)
                Jn = J0 * (torch.exp(P.bv_alpha1 * f * eta) - co / P.bv_c_ref * torch.exp(-P.bv_alpha2 * f * eta))
                if ox < P.m - 1:
                    S[ox + 1] = torch.where(on, -Jn / (P.bv_n * P.F), S[ox + 1])
                S[0] = torch.where(on, -P.z[ox] * Jn / P.bv_n, S[0])
        if self.dirv is not None:
            q, d_ = P.q, self.dim
            off = sum(len(t) for t in P.tags[:2 * a + end])
            g = self.dirv[:, off:off + len(P.tags[2 * a + end])]
            g = g.reshape([1, P.m] + others + [1 if i == d_ - 1 - a else q for i in range(d_)])
            delta = P.C_IP * P.p ** 2 / self.diagonal(a, ha)
            dirich = tag == DIRICHLET
            kappa = sum(kc[k] * c[:, k + 1] for k in range(P.m - 1))
            T0 = S0 = 0.0
            for k in range(P.m - 1):
                f = k + 1
                jc, qn = c[:, f] - g[:, f], un - mig[k] * d[:, 0]
                s = (-D[k] * d[:, f] + D[k] * delta * jc + 0.5 * (c[:, f] + g[:, f]) * qn
                     + 0.5 * torch.abs(qn) * jc)
                S[f], T[f] = torch.where(dirich, s, S[f]), torch.where(dirich, -D[k] * jc, T[f])
                T0, S0 = T0 - ak[k] * jc, S0 - ak[k] * d[:, f]
            jphi = c[:, 0] - g[:, 0]
            S[0] = torch.where(dirich, S0 - kappa * d[:, 0] + delta * kappa * jphi, S[0])
            T[0] = torch.where(dirich, T0 - kappa * jphi, T[0])
        S, T = torch.stack(S, 1) * w, torch.stack(T, 1) * w
        return self.lift(S, sc * T, a, end)

    def __call__(self, U, frozen=None):
        """R(U); with `frozen`, the neighbours' states on every face are taken from it."""
        out, X = self.volume(U), U if frozen is None else frozen
        for a in range(self.dim):
            pos, n = U.dim() - 1 - a - self.dim, U.shape[U.dim() - 1 - a - self.dim]
            cut = lambda t, i, k: t.narrow(pos, i, k)  # noqa: E731
            parts = [self.boundary(a, 0, cut(U, 0, 1)), self.boundary(a, 1, cut(U, n - 1, 1))]
            lower = upper = None
            if n > 1:
                hl, hu = self.h[a][:-1], self.h[a][1:]
                lower, upper = self.interior(a, cut(U, 0, n - 1), cut(X, 1, n - 1), hl, hu)
                if frozen is not None:
                    upper = self.interior(a, cut(X, 0, n - 1), cut(U, 1, n - 1), hl, hu)[1]
            out = out + torch.cat([parts[0]] + ([upper] if n > 1 else []), pos)
            out = out + torch.cat(([lower] if n > 1 else []) + [parts[1]], pos)
        return out

    def jvp(self, u, v):
        return torch.func.jvp(self, (u,), (v,))[1]

    def blocks(self, U):
        """Element-diagonal blocks [batch, E, nb, nb], column by column."""
        P = self.P
        nb = P.m * P.Np
        D = torch.empty(self.batch, P.E, nb, nb, device="cuda", dtype=torch.float64)
        for j in range(nb):
            v = torch.zeros(self.batch, P.m, P.E, P.Np, device="cuda", dtype=torch.float64)
            v[:, j // P.Np, :, j % P.Np] = 1
            col = torch.func.jvp(lambda t: self(t, U), (U,), (v.reshape(self.shape),))[1]
            D[:, :, :, j] = col.reshape(self.batch, P.m, P.E, P.Np).transpose(1, 2).reshape(self.batch, P.E, nb)
        return D


def _by_element(P, x, batch):
    return x.reshape(batch, P.m, P.E, P.Np).transpose(1, 2).reshape(batch, P.E, P.m * P.Np)


def _by_field(P, y, batch):
    return y.reshape(batch, P.E, P.m, P.Np).transpose(1, 2).reshape(-1)


def _sweep(N, U, D, x):
    """(block diagonal + couplings to the element below along x)^-1 x, plane by plane."""
    P, B = N.P, N.batch
    nx = P.n_el[0]
    sel = torch.arange(P.E, device="cuda").reshape(-1, nx)
    xe, z = _by_element(P, x, B), []
    size = [B, P.m] + N.grid[:-1] + [1] + [P.p + 1] * 3
    pos = U.dim() - 4
    to_el = lambda t: t.reshape(B, P.m, -1, P.Np).transpose(1, 2).reshape(B, -1, P.m * P.Np)  # noqa: E731
    for k in range(nx):
        r = xe[:, sel[:, k]]
        if k:
            hl, hu = N.h[0][k - 1:k], N.h[0][k:k + 1]
            zup = z[-1].reshape(B, -1, P.m, P.Np).transpose(1, 2).reshape(size)
            up = torch.func.jvp(lambda t: N.interior(0, t, U.narrow(pos, k, 1), hl, hu)[1],
                                (U.narrow(pos, k - 1, 1),), (zup,))[1]
            r = r - to_el(up)
        z.append(torch.linalg.solve(D[:, sel[:, k]], r.unsqueeze(-1)).squeeze(-1))
    y = torch.empty_like(xe)
    for k in range(nx):
        y[:, sel[:, k]] = z[k]
    return y


def _coarse(N, U, x):
    """The coarse potential correction: one multigrid V-cycle on the element means."""
    P, B = N.P, N.batch
    nz, ny, nx = N.grid
    ix, iy, iz = (torch.arange(P.E, device="cuda") % nx, torch.arange(P.E, device="cuda") // nx % ny,
                  torch.arange(P.E, device="cuda") // (nx * ny))
    colour = (ix + 2 * iy + 3 * iz) % 7
    A = torch.zeros(B, nz, ny, nx, 7, device="cuda", dtype=torch.float64)
    for c in range(7):
        v = torch.zeros(B, P.m, P.E, P.Np, device="cuda", dtype=torch.float64)
        v[:, 0, colour == c] = 1
        s = N.jvp(U, v.reshape(N.shape)).reshape(B, P.m, P.E, P.Np)[:, 0].sum(-1)
        d = (c - colour) % 7
        for k, (off, ok) in enumerate(((0, ix >= 0), (6, ix > 0), (1, ix < nx - 1), (5, iy > 0),
                                       (2, iy < ny - 1), (4, iz > 0), (3, iz < nz - 1))):
            on = ((d == off) & ok).reshape(nz, ny, nx)
            A[..., k] = torch.where(on, s.reshape(B, nz, ny, nx), A[..., k])

    def off(A, t):
        o = torch.zeros_like(t)
        o[..., 1:] += A[..., 1:, 1] * t[..., :-1]
        o[..., :-1] += A[..., :-1, 2] * t[..., 1:]
        o[..., 1:, :] += A[..., 1:, :, 3] * t[..., :-1, :]
        o[..., :-1, :] += A[..., :-1, :, 4] * t[..., 1:, :]
        o[:, 1:] += A[:, 1:, ..., 5] * t[:, :-1]
        o[:, :-1] += A[:, :-1, ..., 6] * t[:, 1:]
        return o

    def smooth(A, t, b, order):
        k = [torch.arange(n, device="cuda") for n in t.shape[1:]]
        par = (k[0][:, None, None] + k[1][:, None] + k[2]) % 2
        for c in order:
            t = torch.where((par == c) & (A[..., 0] != 0), (b - off(A, t)) / A[..., 0], t)
        return t

    def halve(t):
        for ax in (1, 2, 3):
            if t.shape[ax] % 2:
                pad = list(t.shape)
                pad[ax] = 1
                t = torch.cat([t, torch.zeros(pad, device="cuda", dtype=t.dtype)], ax)
        s = t.shape
        return t.reshape([s[0], s[1] // 2, 2, s[2] // 2, 2, s[3] // 2, 2] + list(s[4:])).sum((2, 4, 6))

    def aggregate(A):
        k = [torch.arange(n, device="cuda") for n in A.shape[1:4]]
        C = torch.zeros_like(A)
        C[..., 0] = A[..., 0]
        for d, (even, at) in enumerate(((1, k[2]), (0, k[2]), (1, k[1][:, None]), (0, k[1][:, None]),
                                        (1, k[0][:, None, None]), (0, k[0][:, None, None]))):
            outside = (at % 2 == (0 if even else 1)).expand(A.shape[1:4])
            C[..., d + 1] = torch.where(outside, A[..., d + 1], 0.0)
            C[..., 0] += torch.where(outside, 0.0, A[..., d + 1])
        return halve(C)

    def vcycle(A, b):
        n = b[0].numel()
        if n <= 128:
            eye = torch.eye(n, device="cuda", dtype=torch.float64).reshape([n] + list(b.shape[1:]))
            M = torch.stack([(A[i:i + 1, ..., 0] * eye + off(A[i:i + 1].expand([n] + list(A.shape[1:])), eye)).reshape(n, n).T
                             for i in range(b.shape[0])])
            return torch.linalg.solve(M, b.reshape(b.shape[0], n, 1)).reshape(b.shape)
        t = smooth(A, torch.zeros_like(b), b, (0, 1, 0, 1))
        c = vcycle(aggregate(A), halve(b - A[..., 0] * t - off(A, t)))
        for ax in (1, 2, 3):
            c = c.repeat_interleave(2, ax).narrow(ax, 0, b.shape[ax])
        return smooth(A, t + 1.8 * c, b, (1, 0, 1, 0))

    b = x.reshape(B, P.m, P.E, P.Np)[:, 0].sum(-1).reshape(B, nz, ny, nx)
    return vcycle(A, b).reshape(B, P.E)


def exact(case, seed):
    kind, batch = case["kind"], case.get("batch", 1)
    if kind == "newton":  # its result is the root of R: an iteration of its own would be needed
        return None
    P = _problem(case, seed)
    if kind == "precond_f32" and case["nx"] * case["ny"] * case["nz"] * batch * P.m * P.Np * P.m * P.Np > 6e8:
        return None
    u, v, w, rnd = _inputs(P, case, seed)
    src, dirv = _boundary_data(P, rnd) if kind == "quads" else (None, None)
    N = _Dense(P, batch, src, dirv)
    if kind == "jvp_f32":
        u, v = u.float().double(), v.float().double()
    U, V, W = N.split(u), N.split(v), N.split(w)
    flat = lambda t: t.reshape(-1)  # noqa: E731
    if kind == "quads":
        return flat(N(U)), flat(N.jvp(U, V))
    if kind in ("jvp_df", "jvp_f32"):
        return flat(N.jvp(U, V))
    if kind == "ops_f64":
        return flat(N(U)), flat(N.jvp(U, V)), flat(torch.func.vjp(N, U)[1](W)[0])
    if kind == "grad_df":
        U = U.clone().requires_grad_(True)
        N.theta = {k: t.clone().requires_grad_(True) for k, t in N.theta.items()}
        r = N(U)
        g = torch.autograd.grad(r, [U, N.theta["D"], N.theta["cin"], N.theta["phi"]], W)
        # theta: D_1..D_m, c_in of the unknown species, the applied potentials (which
        # are the handle's own: one value per electrode, summed over the points)
        return flat(r.detach()), flat(g[0]), torch.cat([g[1], g[2][:P.m - 1], g[3].sum(0)])
    x = v.float().double()
    D = N.blocks(U)
    if kind == "precond_f32" and case["nx"] >= 128:
        y = _sweep(N, U, D, x)
    else:
        xe = _by_element(P, x, batch)
        y = torch.cat([torch.linalg.solve(D[:, i:i + 4096], xe[:, i:i + 4096].unsqueeze(-1)).squeeze(-1)
                       for i in range(0, P.E, 4096)], 1)
    y = _by_field(P, y, batch)
    if kind == "precond_f32":
        y = y.reshape(batch, P.m, P.E, P.Np).clone()
        y[:, 0] += _coarse(N, U, x).unsqueeze(-1)
        y = y.reshape(-1)
    return y
