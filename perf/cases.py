"""The work that users of the IBDL library have it do, as cases to time and compare.

Each case goes through the package's public wrappers (``Geometry``, ``Batch``): operator
applications (the step of every GMRES iteration), whole solves, the boundary derivatives of the
backward pass, the field and its post-processing, and batches of small problems. Sizes come from
the workloads of this repository (64² circle, 512² Stokes star, 256 ellipses, 128³ sphere, the
size sweep to 8192², the 1024² differentiation star, the paper's circle study).

Geometries use the library's default launch shapes (no autotuning), in boxes of side 1.
``exact`` restates the operators in 64-bit torch (index_add spreads and torch.fft) without the
package, and solves with a plain GMRES.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2210_07403_gb300.ibdl import Batch, Geometry

# density and data components, and grid fields in and out of the Fourier stage, per equation
_NCOMP = {"scalar": 1, "stokes": 2}


# ------------------------------------------------------------------------------------------
# cases
# ------------------------------------------------------------------------------------------
def _case(do, **kw):
    c = dict(do=do, dim=2, n=512, points=800, curve="star", pde="scalar", lam=0.0, precision="fp64", delta="cos",
             dipole="analytic", symbol="spectral")
    c.update(kw)
    return c


def listed():
    return [
        # the smallest problem: one FP64 application on the 64² circle (latency and launches)
        _case("apply", name="apply_circle_64_fp64", n=64, points=100, curve="circle"),
        # the Stokes star at 512²: the FP64 application of plain solves and of FP64 residuals …
        _case("apply", name="apply_star_512_fp64", pde="stokes"),
        # … the FP32 application of the inner iterations of mixed solves …
        _case("apply", name="apply_star_512_fp32", pde="stokes", precision="fp32"),
        # … and the whole mixed-precision solve that both serve
        _case("solve", name="solve_star_512_mixed", pde="stokes", precision="mixed"),
        # the paper's own discretisation (finite differences, √ delta, divergence of the spread
        # vector) on its circle study's finest grid
        _case("apply", name="apply_paper_circle_2048_fp64", n=2048, points=4289, curve="circle", lam=1.0, delta="sqrt",
              dipole="spectral_div", symbol="fd2"),
        # the largest grid: bound by HBM traffic
        _case("apply", name="apply_circle_8192_fp32", n=8192, points=17157, curve="circle", precision="fp32"),
        # many independent problems of 128² … 512² at once: one batched FP32 application …
        _case("batch_apply", name="batch_apply_ellipses_256_fp32", count=256, n=512, curve="ellipse", precision="fp32"),
        # … and a batched mixed-precision solve
        _case("batch_solve", name="batch_solve_ellipses_64_mixed", count=64, n=512, curve="ellipse", precision="mixed"),
        # the 3-D sphere: an FP64 application and the whole mixed-precision solve
        _case("apply", name="apply_sphere_128_fp64", dim=3, n=128, points=12000, curve="sphere"),
        _case("solve", name="solve_sphere_128_mixed", dim=3, n=128, points=12000, curve="sphere", precision="mixed"),
        # the backward pass of a shape objective: derivatives to X, n and Δs of the 1024² Stokes star
        _case("vjp", name="vjp_star_1024_fp64", n=1024, points=1600, pde="stokes"),
        # after a solve: the field on the grid, the indicator of the domain and the interpolation of
        # the values near the boundary (the paper's spectral settings)
        _case("post", name="post_circle_1024_fp64", n=1024, points=2145, curve="circle"),
    ]


def draw(rng):
    def size(lo, hi):  # a power of two in [lo, hi], uniform in its logarithm
        return 2 ** rng.randint(int(math.log2(lo)), int(math.log2(hi)))

    def points(n):  # boundary points at Δs ≈ 0.5h … 1.5h on a curve of length about 1.5
        return max(8, int(1.5 * n / rng.uniform(0.5, 1.5)))

    do = rng.choice(["apply", "apply", "apply", "transpose", "solve", "batch_apply", "batch_solve", "vjp", "post", "sphere"])
    opts = dict(delta=rng.choice(["cos", "sqrt"]), symbol=rng.choice(["spectral", "fd2"]))
    lam = rng.choice([0.0, rng.uniform(0.1, 100.0)])
    curve = rng.choice(["circle", "star", "ellipse"])
    if do == "sphere":
        n = size(16, 128)
        precision = rng.choice(["fp64", "fp32", "mixed"])
        return _case("solve" if precision == "mixed" else "apply", dim=3, n=n, curve="sphere", lam=lam,
                     points=int(0.75 * n * n * rng.uniform(0.5, 1.0)) + 8, precision=precision, **opts)
    pde = rng.choice(["scalar", "stokes"])
    if do in ("batch_apply", "batch_solve"):
        count = int(2 ** rng.uniform(1, 8 if do == "batch_apply" else 6))
        precision = rng.choice(["fp32", "fp64"]) if do == "batch_apply" else "mixed"
        n = 512 if precision != "fp64" else 256
        return _case(do, count=count, n=n, curve="ellipse", precision=precision, **opts)
    if do == "solve":
        n = size(64, 512)
        return _case(do, n=n, points=int(1.5 * n / rng.uniform(0.75, 1.25)), curve=curve, pde=pde,
                     lam=lam if pde == "scalar" else 0.0, precision=rng.choice(["mixed", "fp64"]), symbol="spectral")
    if do == "vjp":
        n = size(64, 1024)
        return _case(do, n=n, points=points(n), curve=curve, pde=pde, lam=lam, symbol=opts["symbol"])
    if do == "post":
        n = size(64, 1024)
        return _case(do, n=n, points=points(n), curve=curve, lam=lam, **opts)
    precision = rng.choice(["fp64", "fp32", "fp32x2"])
    dipole = "analytic" if pde == "stokes" and do == "transpose" else rng.choice(["analytic", "analytic", "spectral_div"])
    n = size(16, {"fp64": 2048, "fp32": 8192 if pde == "scalar" else 4096, "fp32x2": 2048}[precision])
    return _case(do, n=n, points=points(n), curve=curve, pde=pde, lam=lam, precision=precision, dipole=dipole, **opts)


# ------------------------------------------------------------------------------------------
# boundaries and data from a seed
# ------------------------------------------------------------------------------------------
def _curve(radius, M, centre, rot):
    """Star-shaped curve r(θ), M points equispaced in arclength, outward normals, weights Δs."""
    th = np.linspace(0.0, 2 * np.pi, 16385)
    r = radius(th)
    x, y = r * np.cos(th), r * np.sin(th)
    s = np.concatenate([[0.0], np.cumsum(np.hypot(np.diff(x), np.diff(y)))])
    t = np.interp(s[-1] * np.arange(M) / M, s, th)
    e = 1e-5
    r, dr = radius(t), (radius(t + e) - radius(t - e)) / (2 * e)
    tx, ty = dr * np.cos(t) - r * np.sin(t), dr * np.sin(t) + r * np.cos(t)
    sp = np.hypot(tx, ty)
    c, q = math.cos(rot), math.sin(rot)
    R = np.array([[c, -q], [q, c]])
    X = np.asarray(centre)[:, None] + R @ np.stack([r * np.cos(t), r * np.sin(t)])
    n = R @ np.stack([ty / sp, -tx / sp])
    return X, n / np.sqrt(np.sum(n * n, axis=0)), np.full(M, s[-1] / M)


def _boundary(curve, M, h, g, i):
    """The curve or surface about the box's middle, moved by up to half a cell. Ellipse i of a batch
    has the same semi-axes (and so the same number of points) for every seed."""
    if curve == "sphere":
        k = np.arange(M)
        z = 1 - (2 * k + 1) / M
        rho, ph = np.sqrt(1 - z * z), k * np.pi * (3 - math.sqrt(5))
        n = np.stack([rho * np.cos(ph), rho * np.sin(ph), z])
        X = 0.5 + h * g.uniform(-0.5, 0.5, size=(3, 1)) + 0.25 * n
        return X, n / np.sqrt(np.sum(n * n, axis=0)), np.full(M, 4 * np.pi * 0.25 ** 2 / M)
    centre = 0.5 + h * g.uniform(-0.5, 0.5, size=2)
    if curve == "circle":
        return _curve(lambda t: 0.25 + 0.0 * t, M, centre, g.uniform(0, 2 * np.pi))
    if curve == "star":
        return _curve(lambda t: 0.25 * (1 + 0.2 * np.cos(5 * t)), M, centre, 0.0)
    a, b = np.random.default_rng([i, 3]).uniform(0.1, 0.3, size=2)
    radius = lambda t: 1.0 / np.sqrt((np.cos(t) / a) ** 2 + (np.sin(t) / b) ** 2)  # noqa: E731
    if M is None:  # Δs ≈ h
        M = max(8, int(round(_curve(radius, 8, centre, 0.0)[2].sum() / h)))
    return _curve(radius, M, centre, g.uniform(0, np.pi))


def _smooth(X, c, g, K=8):
    """Smooth random boundary data: modes |m| ≤ K of the angle about the box's middle ([c][M])."""
    t = np.arctan2(X[1] - 0.5, X[0] - 0.5)
    m = np.arange(K + 1)
    out = np.zeros((c, X.shape[1]))
    for l in range(c):
        a, b = g.standard_normal((2, K + 1)) / np.sqrt(2 * K + 1)
        out[l] = np.cos(np.outer(t, m)) @ a + np.sin(np.outer(t, m)) @ b
    if X.shape[0] == 3:
        out *= 1 + X[2] - 0.5
    return out


def _problems(case, seed):
    """Plain descriptions of the case's problem, or of the problems of its batch."""
    g = np.random.default_rng([seed, 2210])
    out = []
    for i in range(case.get("count", 1)):
        batch = "count" in case
        n = case["n"] // (4 >> (i % 3)) if batch else case["n"]  # a batch holds n/4, n/2 and n in turn
        X, nrm, w = _boundary(case["curve"], None if batch else case["points"], 1.0 / n, g, i)
        lam = float(g.uniform(0, 100)) if batch else case["lam"]
        c = _NCOMP[case["pde"]]
        data = _smooth(X, c, g, 6 if batch else 8)
        if case["pde"] == "stokes" and case["do"] == "solve":  # interior Stokes data carry no flux
            data = data - (np.sum(w * data * nrm) / np.sum(w)) * nrm
        if case["do"] in ("apply", "batch_apply", "transpose", "vjp"):  # densities as in a Krylov space
            data = data + 0.1 * g.standard_normal(data.shape)
        out.append(SimpleNamespace(N=n, box=1.0, origin=(0.0, 0.0, 0.0), pde=case["pde"], lam=lam, mu=1.0,
                                   delta=case["delta"], dipole=case["dipole"], symbol=case["symbol"],
                                   bd=SimpleNamespace(X=X, n=nrm, w=w), data=data.reshape(-1),
                                   other=(_smooth(X, c, g) + 0.1 * g.standard_normal((c, X.shape[1]))).reshape(-1)))
    return out


def prepare(case, seed):
    ps = _problems(case, seed)
    if "count" in case:
        handle = Batch(ps)
    else:
        handle = Geometry.from_problem(ps[0])
    s = SimpleNamespace(do=case["do"], precision=case["precision"], n=case["n"], h=handle,
                        v=torch.from_numpy(np.concatenate([p.data for p in ps])).cuda())
    if case["do"] == "vjp":
        s.other = torch.from_numpy(ps[0].other).cuda()
    return s


# ------------------------------------------------------------------------------------------
# one pass
# ------------------------------------------------------------------------------------------
RTOL = 1e-10  # of the solves


def run(s):
    if s.do in ("apply", "batch_apply"):
        return s.h.apply(s.v, precision=s.precision)
    if s.do == "transpose":
        return s.h.apply_transpose(s.v, precision=s.precision)
    if s.do in ("solve", "batch_solve"):
        return s.h.solve(s.v, rtol=RTOL, precision=s.precision, maxit=400)[0]
    if s.do == "vjp":
        return s.h.solve_vjp(s.v, s.other)
    u = s.h.evaluate_field(s.v)
    chi, flags = s.h.indicator()
    m1 = 2.0 * (math.log2(s.n) - 4.0)
    return {"u": u, "chi": chi, "flags": flags, "near": s.h.near_boundary(s.v, u, flags, m1, m1 + 2.0)}


def work(case):
    """Boundary data and results moved once; 2.5 N log₂ N operations per real transform of N nodes
    and 5 per node and field for the symbol. Solves: their usual number of applications."""
    total = {"bytes": 0.0, "flops": 0.0}
    for i in range(case.get("count", 1)):
        n, dim, c = case["n"] // (4 >> (i % 3)) if "count" in case else case["n"], case["dim"], _NCOMP[case["pde"]]
        M = int(1.25 * n) if "count" in case else case["points"]
        fields = 2 if case["pde"] == "scalar" else 5
        if case["dipole"] == "spectral_div":
            fields += 1
        nodes = float(n) ** dim
        apply = nodes * fields * (2.5 * dim * math.log2(n) + 5.0)
        point = 8.0 * M * (2 * dim + 1)
        if case["do"] in ("solve", "batch_solve"):
            total["bytes"] += point + 16.0 * M * c
            total["flops"] += apply * (30 if case["pde"] == "stokes" else 14)
        elif case["do"] == "vjp":
            total["bytes"] += 2 * point + 16.0 * M * c
            total["flops"] += 2 * apply
        elif case["do"] == "post":
            total["bytes"] += point + 8.0 * M + nodes * (8 + 8 + 1 + 8)
            total["flops"] += 2 * apply
        else:
            total["bytes"] += point + 16.0 * M * c
            total["flops"] += apply
    return total


# ------------------------------------------------------------------------------------------
# the same in 64-bit torch
# ------------------------------------------------------------------------------------------
def _phi(r, kind):
    a = r.abs()
    if kind == "cos":
        return torch.where(a < 2, 0.25 * (1 + torch.cos(0.5 * math.pi * r)), torch.zeros_like(r))
    inner = (3 - 2 * a + torch.sqrt((1 + 4 * a - 4 * a * a).clamp_min(0.0))) / 8
    outer = (5 - 2 * a - torch.sqrt((-7 + 12 * a - 4 * a * a).clamp_min(0.0))) / 8
    return torch.where(a <= 1, inner, torch.where(a < 2, outer, torch.zeros_like(r)))


def _dphi(r, kind):
    a = r.abs()
    if kind == "cos":
        return torch.where(a < 2, -0.125 * math.pi * torch.sin(0.5 * math.pi * r), torch.zeros_like(r))
    inner = (-2 + (2 - 4 * a) / torch.sqrt((1 + 4 * a - 4 * a * a).clamp_min(1e-300))) / 8
    outer = (-2 - (6 - 4 * a) / torch.sqrt((-7 + 12 * a - 4 * a * a).clamp_min(1e-300))) / 8
    return torch.sign(r) * torch.where(a <= 1, inner, torch.where(a < 2, outer, torch.zeros_like(r)))


class _Exact:
    """The operators of one problem (X, n and w may carry gradients)."""

    def __init__(self, p, X=None, nrm=None, w=None):
        dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
        self.p, self.X = p, dev(p.bd.X) if X is None else X
        self.n, self.w = dev(p.bd.n) if nrm is None else nrm, dev(p.bd.w) if w is None else w
        self.N, self.dim, self.hh = p.N, self.X.shape[0], 1.0 / p.N
        N, dim = self.N, self.dim
        xi = self.X / self.hh
        base = torch.floor(xi.detach()).long() - 1
        a = torch.arange(4, device="cuda")
        r = (base[:, :, None] + a) - xi[:, :, None]
        idx = (base[:, :, None] + a) % N
        ph, dp = _phi(r, p.delta), _dphi(r, p.delta) / self.hh
        M = self.X.shape[1]

        def outer(f):  # product over the axes of f[j][M][4] → [M][4^dim], x fastest
            v = f[dim - 1]
            for j in range(dim - 2, -1, -1):
                v = (v[:, :, None] * f[j][:, None, :]).reshape(M, -1)
            return v

        lin = idx[dim - 1]
        for j in range(dim - 2, -1, -1):
            lin = (lin[:, :, None] * N + idx[j][:, None, :]).reshape(M, -1)
        self.lin, self.val = lin, outer(ph)
        self.grad = [outer([dp[j] if j == m else ph[j] for j in range(dim)]) for m in range(dim)]
        m = torch.fft.fftfreq(N, d=1.0 / N, dtype=torch.float64, device="cuda")
        k = 2 * math.pi * m
        if p.symbol == "spectral":
            lap1, der1 = k * k, k.clone()
            der1[N // 2] = 0.0
        else:
            lap1, der1 = 4.0 * N * N * torch.sin(0.5 * k / N) ** 2, N * torch.sin(k / N)
        half = N // 2 + 1  # real transforms keep kx = 0 … N/2
        shape = lambda v, j: (v[:half] if j == 0 else v).reshape([-1 if dim - 1 - i == j else 1 for i in range(dim)])  # noqa: E731
        self.lap = sum(shape(lap1, j) for j in range(dim))
        self.der = [shape(der1, j) for j in range(dim)]

    def spread(self, weights):  # weights [M][4^dim] at the stencil's nodes
        f = torch.zeros(self.N ** self.dim, dtype=torch.float64, device="cuda")
        return f.index_add(0, self.lin.reshape(-1), weights.reshape(-1)).reshape((self.N,) * self.dim)

    def fft(self, f):
        return torch.fft.rfftn(f)

    def ifft(self, F):
        return torch.fft.irfftn(F, s=(self.N,) * self.dim)

    def inv(self, den):
        return torch.where(den != 0, 1.0 / torch.where(den != 0, den, torch.ones_like(den)), torch.zeros_like(den))

    def gather(self, u, weights):
        return (u.reshape(-1)[self.lin] * weights).sum(1)

    def scale(self):
        return self.w / self.hh ** self.dim

    def field(self, Q, laplace=False):
        p, s, d = self.p, self.scale(), self.dim
        if p.pde == "scalar" or laplace:
            q = (Q if not laplace else torch.ones_like(self.w)) * s
            if p.dipole == "analytic":
                F = self.fft(self.spread(sum((q * self.n[m])[:, None] * self.grad[m] for m in range(d))))
            else:
                F = sum(1j * self.der[m] * self.fft(self.spread((q * self.n[m])[:, None] * self.val)) for m in range(d))
            return self.ifft(F * self.inv(self.lap + (0.0 if laplace else p.lam)))[None]
        Q = Q.reshape(2, -1)
        S = self.fft(self.spread((s * (Q * self.n).sum(0))[:, None] * self.val))
        A = [[s * (Q[l] * self.n[m] + Q[m] * self.n[l]) for m in range(2)] for l in range(2)]
        if p.dipole == "analytic":
            G = [self.fft(self.spread(sum(A[l][m][:, None] * self.grad[m] for m in range(2)))) for l in range(2)]
        else:
            T = [[self.fft(self.spread(A[l][m][:, None] * self.val)) for m in range(2)] for l in range(2)]
            G = [sum(1j * self.der[m] * T[l][m] for m in range(2)) for l in range(2)]
        inv = self.inv(self.lap)
        kg = sum(self.der[m] * G[m] for m in range(2))
        proj = p.mu * self.inv(p.mu * self.lap + p.lam) if p.lam > 0 else inv
        return torch.stack([self.ifft(1j * self.der[l] * S * inv + (G[l] - self.der[l] * kg * inv) * proj) for l in range(2)])

    def apply(self, Q):
        u = self.field(Q)
        return torch.cat([self.gather(v, self.val) for v in u]) + 0.5 * Q

    def transpose(self, G):
        """Aᵀ G by reverse differentiation of the (linear) application."""
        Q = torch.zeros_like(G, requires_grad=True)
        return torch.autograd.grad(self.apply(Q), Q, G)[0]

    def solve(self, b):
        """GMRES without restarts, modified Gram-Schmidt twice, to a residual of 1e-13."""
        beta = b.norm()
        V, H = [b / beta], torch.zeros(201, 200, dtype=torch.float64)
        for k in range(200):
            w = self.apply(V[k])
            for _ in range(2):
                for i, v in enumerate(V):
                    c = torch.dot(v, w)
                    w = w - c * v
                    H[i, k] += float(c)
            H[k + 1, k] = float(w.norm())
            e = torch.zeros(k + 2, dtype=torch.float64)
            e[0] = float(beta)
            y = torch.linalg.lstsq(H[:k + 2, :k + 1], e[:, None]).solution[:, 0]
            if float((H[:k + 2, :k + 1] @ y - e).norm()) < 1e-13 * float(beta) or k == 199:
                break
            V.append(w / H[k + 1, k].item())
        return sum(float(y[i]) * V[i] for i in range(len(y)))


def exact(case, seed):
    out = []
    for p in _problems(case, seed):
        v = torch.from_numpy(p.data).cuda()
        if case["do"] == "vjp":
            dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda().requires_grad_() for a in (p.bd.X, p.bd.n, p.bd.w)]
            J = -torch.dot(torch.from_numpy(p.other).cuda(), _Exact(p, *dev).apply(v))
            return tuple(torch.autograd.grad(J, dev))
        op = _Exact(p)
        if case["do"] == "post":
            chi = op.field(v, laplace=True)[0]
            chi = chi - chi.reshape(-1)[0]
            return {"u": op.field(v)[0], "chi": chi, "flags": None, "near": None}
        out.append({"transpose": op.transpose, "solve": op.solve, "batch_solve": op.solve}.get(case["do"], op.apply)(v))
    return torch.cat(out)
