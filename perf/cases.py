"""What this repository's speed is measured on: the calls a user of the solver makes, from one plane wave on a
small contour to a thousand on a large one, in both forms.

A case is one call (or one short sequence of calls) through the public Python interface:

* ``solve``     plane waves through a factored context (the daily call: many per setup);
* ``general``   a general right-hand side, forward or adjoint, through a factored context;
* ``pipeline``  contour, mesh, assembly, skeleton, factors and the first plane waves: what a new contour costs;
* ``assemble``  operators of a new mesh and one product with C: what diagnostics and iterative solvers do;
* ``batch``     several contours of uneven size with results on the host;
* ``gradient``  the far-field shape gradient (the optimisation loop's step);
* ``farfield``  far fields of many currents.

The mixed form's results are documented to 1e-6 (the FP64 form's to 1e-10), so a program that keeps them keeps
them in single precision: ``run`` hands the mixed form's blocks on as complex64, the FP64 form's as complex128.
With ``exact_residual`` the mixed form refines to its stored operator, whose entries carry 24 bits: complex64 too.

``exact`` is the same discretisation (Galerkin, linear hats, uniform in arc length) written in plain torch in 64
bits, solved densely.
"""

import math

import numpy as np
import torch

from paper_2203_13283_gb300 import Solver
from paper_2203_13283_gb300.solver import batch_solve_fourier

DENSE_LIMIT = 4200   # largest N that exact() assembles and factors densely


# --------------------------------------------------------------------------- the cases
def listed():
    return [
        # one plane wave on a small contour: every kernel is short, launches and host steps count
        dict(name="solve_fp64_n256_b1", kind="solve", family="ellipse", N=256, B=1, precision=0, rank_div=4),
        # the default (FP64) form in ordinary use: a contour of odd size, a block of incidences
        dict(name="solve_fp64_n1501_b32", kind="solve", family="star", N=1501, B=32, precision=0, rank_div=8),
        # the 360-incidence ellipse: mixed form, a monostatic sweep at one-degree steps
        dict(name="solve_mixed_n4096_b360", kind="solve", family="ellipse", N=4096, B=360, precision=1, rank_div=8),
        # the largest: 1024 incidences on the superellipse
        dict(name="solve_mixed_n16384_b1024", kind="solve", family="superellipse", N=16384, B=1024, precision=1,
             rank_div=8, chunk=1024),
        # refinement to the stored operator with exact residuals
        dict(name="solve_exact_n4096_b64", kind="solve", family="superellipse", N=4096, B=64, precision=1, rank_div=8,
             exact_residual=1),
        # backward pass of the autograd wrapper: adjoint solve of a general block, odd N
        dict(name="adjoint_mixed_n3001_b24", kind="general", family="star", N=3001, B=24, precision=1, rank_div=8,
             adjoint=True),
        # a new contour from its coefficients to its first currents, mixed form, ragged size
        dict(name="pipeline_mixed_n2777_b64", kind="pipeline", family="star", N=2777, B=64, precision=1, rank_div=8),
        # the same in the default form
        dict(name="pipeline_fp64_n1024_b8", kind="pipeline", family="ellipse", N=1024, B=8, precision=0, rank_div=8),
        # operators of a larger mesh and one product with C
        dict(name="assemble_mixed_n8192_b16", kind="assemble", family="superellipse", N=8192, B=16, precision=1),
        # many contours of uneven size, as the batched form is used
        dict(name="batch_mixed_6x64", kind="batch", count=6, n_min=512, n_max=4096, B=64, precision=1, rank_div=8),
        # one step of a shape optimisation
        dict(name="gradient_fp64_n1024_m4", kind="gradient", family="ellipse", N=1024, B=8, nphi=45, M=4, precision=0,
             rank_div=4),
        # far fields of a block of currents over the full circle
        dict(name="farfield_n16384_b256_o360", kind="farfield", family="superellipse", N=16384, B=256, nphi=360,
             precision=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "general", "pipeline", "pipeline", "assemble", "batch", "gradient",
                       "farfield"])
    family = rng.choice(["ellipse", "superellipse", "star"])
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(2, 6), n_min=_log_int(rng, 200, 600), n_max=_log_int(rng, 1000, 4096),
                    B=_log_int(rng, 4, 64), precision=1, rank_div=8)
    if kind == "gradient":
        # (a superellipse has points of zero curvature: the perturbed contours of its gradient are not convex)
        return dict(kind="gradient", family=rng.choice(["ellipse", "star"]), N=_log_int(rng, 150, 1100), B=rng.randint(1, 12),
                    nphi=_log_int(rng, 8, 90), M=rng.randint(1, 4), precision=0, rank_div=4)
    if kind == "farfield":
        return dict(kind="farfield", family=family, N=_log_int(rng, 300, 16384), B=_log_int(rng, 1, 256),
                    nphi=_log_int(rng, 16, 360), precision=0)
    precision = rng.choice([0, 1, 1])
    if kind == "assemble":
        return dict(kind="assemble", family=family, N=_log_int(rng, 300, 8192 if precision else 1600),
                    B=_log_int(rng, 1, 32), precision=precision)
    if kind == "pipeline":
        return dict(kind="pipeline", family=family, N=_log_int(rng, 200, 5000 if precision else 1100),
                    B=_log_int(rng, 1, 64), precision=precision, rank_div=8)
    case = dict(kind=kind, family=family, N=_log_int(rng, 200, 6000 if precision else 1600),
                B=_log_int(rng, 1, 400 if precision else 48), precision=precision, rank_div=8)
    if kind == "general":
        case["adjoint"] = rng.random() < 0.5
    elif precision and rng.random() < 0.25:
        case.update(exact_residual=1, N=_log_int(rng, 300, 4096), B=_log_int(rng, 1, 64))
    return case


# --------------------------------------------------------------------------- inputs
def _star(rng):
    """Coefficients of a convex star r = 1 + sum a_m cos(m theta + phi_m), a_m ~ U(0, 0.02 / m^2)."""
    c, s = np.zeros(9), np.zeros(9)
    c[0] = 1.0
    for m in range(2, 9):
        a, ph = rng.uniform(0.0, 0.02 / m ** 2), rng.uniform(0.0, 2.0 * math.pi)
        c[m], s[m] = a * math.cos(ph), -a * math.sin(ph)
    return c, s


def _contour(family, rng):
    if family == "ellipse":
        return "ellipse", dict(ax=1.0, ay=float(rng.uniform(0.45, 0.8)))
    if family == "superellipse":
        return "superellipse", dict(ax=1.0, ay=float(rng.uniform(0.55, 0.8)), p=4.0)
    c, s = _star(rng)
    return "fourier", dict(cos=c, sin=s)


def _inputs(case, seed):
    """The user's data of a case: contour, angles, blocks (numpy, from the seed alone)."""
    rng = np.random.default_rng(seed)
    d = {}
    if case["kind"] == "batch":
        lo, hi, last = case["n_min"], case["n_max"], max(1, case["count"] - 1)
        n = [int(lo * (hi / lo) ** (i / last)) for i in range(case["count"])]
        d["contours"] = []
        for ni in n:
            c, s = _star(rng)
            d["contours"].append(dict(cos=c.tolist(), sin=s.tolist(), N=int(ni)))
    else:
        d["family"], d["params"] = _contour(case["family"], rng)
    B = case["B"]
    d["angles"] = rng.uniform(0.0, 2.0 * math.pi) + 2.0 * math.pi * np.arange(B) / B
    if "nphi" in case:
        d["phi"] = rng.uniform(0.0, 0.1) + 2.0 * math.pi * np.arange(case["nphi"]) / case["nphi"]
    d["seed"] = int(rng.integers(1, 1 << 30))
    return d


def _block(case, d):
    """A block of smooth currents: each column a few Fourier modes of the propagating range (amplitude ~1), N x B on the GPU."""
    N, B = case["N"], case["B"]
    g = torch.Generator(device="cuda").manual_seed(d["seed"])
    hat = torch.zeros((B, N), dtype=torch.complex128, device="cuda")
    w = max(2, N // 10)
    z = torch.randn((2, B, 2 * w), dtype=torch.float64, device="cuda", generator=g)
    z = torch.complex(z[0], z[1]) / math.sqrt(4.0 * w)
    hat[:, :w], hat[:, N - w:] = z[:, :w], z[:, w:]
    return (torch.fft.ifft(hat, dim=1) * N).t()   # N x B, columns contiguous


def _solver(case, d):
    opt = dict(precision=case["precision"])
    if case["precision"]:
        # the drained residual of a general block floors above a plane wave's
        opt["refine_tol"] = 1e-6 if case["kind"] == "general" else 5e-7
    if case.get("exact_residual"):
        opt.update(exact_residual=1, refine_tol=1e-10)
    if "chunk" in case:
        opt["rhs_chunk"] = case["chunk"]
    return Solver(**opt).contour(d["family"], **d["params"])


def _factor(s, case, d):
    s.mesh(case["N"]).assemble()
    s.skeleton(1e-6, max_rank=max(16, case["N"] // case["rank_div"]), seed=d["seed"], allow_cap=True)
    return s.factor()


def prepare(case, seed):
    d = _inputs(case, seed)
    st = dict(case=case, d=d)
    if case["kind"] == "batch":
        return st
    st["s"] = s = _solver(case, d)
    if case["kind"] in ("solve", "general", "gradient"):
        _factor(s, case, d)
    elif case["kind"] == "farfield":
        s.mesh(case["N"])
    if case["kind"] in ("general", "assemble", "farfield"):
        st["x"] = _block(case, d)
    return st


# --------------------------------------------------------------------------- one pass
def run(st):
    case, d, s = st["case"], st["d"], st.get("s")
    kind = case["kind"]
    if kind == "batch":
        js, _ = batch_solve_fourier(d["contours"], d["angles"], tol=1e-6, rank_div=case["rank_div"], workers=2,
                                    precision=case["precision"], refine_tol=5e-7)
        return [j.astype(np.complex64) for j in js]
    if kind == "gradient":
        return list(s.shape_gradient(d["angles"], d["phi"], case["M"]))
    if kind == "farfield":
        return s.farfield(st["x"], d["phi"])
    if kind == "solve":
        out = s.solve_planewaves(d["angles"])
    elif kind == "general":
        out = s.solve_adjoint(st["x"]) if case["adjoint"] else s.solve(st["x"])
    elif kind == "pipeline":
        s.contour(d["family"], **d["params"])
        out = _factor(s, case, d).solve_planewaves(d["angles"])
    else:
        s.contour(d["family"], **d["params"]).mesh(case["N"]).assemble()
        out = s.apply("C", st["x"])
    return out.to(torch.complex64) if case["precision"] else out


# --------------------------------------------------------------------------- what a pass cannot do without
def _entry_bytes(case):
    return 12 if case["precision"] else 16   # three bf16 planes of (re, im), or complex FP64


def _assemble_work(N, eb):
    # one evaluation of two Hankel orders at two wavenumbers for 16 point pairs of each element pair, ~40 flops each
    return 4.0 * N * N * eb, 16.0 * 4.0 * 40.0 * N * N


def _solve_work(case, N, B):
    # the right-hand side, Eq. (9) and one residual: six operator products and the two Woodbury ones; operators and factors read once
    eb, r = _entry_bytes(case), max(16, N // case["rank_div"])
    return 4.0 * N * N * eb + 32.0 * N * r + 16.0 * N * B, 8.0 * B * (6.0 * N * N + 2.0 * N * r)


def _setup_work(case, N):
    # assembly; r samples and r rows of V^T (four products each), the projections, K and its inverse
    b, f = _assemble_work(N, _entry_bytes(case))
    r = max(16, N // case["rank_div"])
    return b + 3 * 16.0 * N * r, f + 8.0 * (8.0 * N * N * r + 4.0 * N * r * r + 2.0 * r ** 3)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        b = f = 0.0
        for i in range(case["count"]):
            n = case["n_min"] * (case["n_max"] / case["n_min"]) ** (i / max(1.0, case["count"] - 1.0))
            w = work(dict(case, kind="pipeline", N=int(n)))
            b, f = b + w["bytes"], f + w["flops"]
        return dict(bytes=b, flops=f)
    N, B = case["N"], case["B"]
    if kind in ("solve", "general"):
        b, f = _solve_work(case, N, B)
    elif kind == "pipeline":
        (b, f), (b2, f2) = _setup_work(case, N), _solve_work(case, N, B)
        b, f = b + b2, f + f2
    elif kind == "assemble":
        b, f = _assemble_work(N, _entry_bytes(case))
        b, f = b + 32.0 * N * B, f + 8.0 * 4.0 * N * N * B
    elif kind == "gradient":
        b, f = _solve_work(case, N, 2 * B)
        b, f = b + 64.0 * N * N, f + 36.0 * 4.0 * 80.0 * N * N + 8.0 * 4.0 * N * N * B
    else:
        q = 12.0   # one exponential (~40 flops) per quadrature point and direction, one product with the currents
        b, f = 16.0 * N * B + 16.0 * case["nphi"] * B, case["nphi"] * N * (8.0 * B + 40.0 * q)
    return dict(bytes=b, flops=f)


# --------------------------------------------------------------------------- the same in 64 bits, plain torch
def _gauss01(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return 0.5 * (x + 1.0), 0.5 * w


def _radial(family, p, th):
    """rho, rho', rho'' of the contour r = rho(theta) (cos, sin)."""
    c, s = torch.cos(th), torch.sin(th)
    if family == "fourier":
        r, r1, r2 = (torch.zeros_like(th) for _ in range(3))
        for m, (a, b) in enumerate(zip(p["cos"], p["sin"])):
            cm, sm = torch.cos(m * th), torch.sin(m * th)
            r, r1, r2 = r + a * cm + b * sm, r1 + m * (b * cm - a * sm), r2 - m * m * (a * cm + b * sm)
        return r, r1, r2
    q = 2.0 if family == "ellipse" else p["p"]
    u, v = (c / p["ax"]).abs(), (s / p["ay"]).abs()
    su, sv = torch.sign(c) / p["ax"], torch.sign(s) / p["ay"]
    # f = u^q + v^q, rho = f^(-1/q); du/dtheta = -sign(c) s / ax, dv/dtheta = sign(s) c / ay
    du, dv = -su * s, sv * c
    f = u ** q + v ** q
    f1 = q * (u ** (q - 1) * du + v ** (q - 1) * dv)
    f2 = q * ((q - 1) * (u ** (q - 2) * du ** 2 + v ** (q - 2) * dv ** 2) - u ** q - v ** q)
    r = f ** (-1.0 / q)
    r1 = -r * f1 / (q * f)
    r2 = -(r1 * f1 + r * f2) / (q * f) + r * f1 ** 2 / (q * f ** 2)
    return r, r1, r2


class _Mesh:
    """Points of the arc-length-uniform mesh."""

    def __init__(self, family, params, N, dev):
        self.family, self.params, self.N, self.dev = family, params, N, dev
        P = 4096
        x, w = _gauss01(20)
        self.x, self.w = (torch.tensor(v, dtype=torch.float64, device=dev) for v in (x, w))
        self.edge = torch.arange(P + 1, dtype=torch.float64, device=dev) * (2.0 * math.pi / P)
        self.step = 2.0 * math.pi / P
        part = self._length(self.edge[:-1], self.edge[1:])
        self.cum = torch.cat([torch.zeros(1, dtype=torch.float64, device=dev), torch.cumsum(part, 0)])
        self.L = float(self.cum[-1])
        self.h = self.L / N
        self.k = 2.0 * math.pi * (N / 10.0) / self.L
        self.a = self.L / (2.0 * math.pi)
        self.kt = complex(self.k, 0.4 * self.k ** (1.0 / 3.0) * self.a ** (-2.0 / 3.0))

    def _speed(self, th):
        r, r1, _ = _radial(self.family, self.params, th)
        return torch.sqrt(r * r + r1 * r1)

    def _length(self, t0, t1):
        d = t1 - t0
        return (self._speed(t0[:, None] + d[:, None] * self.x) * self.w).sum(1) * d

    def points(self, xi):
        """(N, q) x, y, nx, ny, curvature at local coordinates xi of every element."""
        s = ((torch.arange(self.N, dtype=torch.float64, device=self.dev)[:, None] + xi) * self.h).reshape(-1)
        i = (torch.searchsorted(self.cum, s, right=True) - 1).clamp(0, len(self.cum) - 2)
        th = self.edge[i] + self.step * (s - self.cum[i]) / (self.cum[i + 1] - self.cum[i])
        for _ in range(6):
            th = th - (self.cum[i] + self._length(self.edge[i], th) - s) / self._speed(th)
        r, r1, r2 = _radial(self.family, self.params, th)
        c, sn = torch.cos(th), torch.sin(th)
        tx, ty = r1 * c - r * sn, r1 * sn + r * c
        v = torch.sqrt(tx * tx + ty * ty)
        kap = (r * r + 2.0 * r1 * r1 - r * r2) / v ** 3
        return [t.reshape(self.N, -1) for t in (r * c, r * sn, ty / v, -tx / v, kap)]


def _hankel(x, kp):
    """H0, H1, J0, J1 at z = x (1 + i kp) for real x (flat tensor), J only below x = 5."""
    out = [torch.zeros_like(x, dtype=torch.complex128) for _ in range(4)]
    big, far = x >= 25.0, (x > 5.0) & (x < 25.0)
    z = x[big] * complex(1.0, kp)
    if z.numel():
        # Hankel's expansion
        w, amp = 1j / z, torch.sqrt(2.0 / (math.pi * z)) * torch.exp(1j * (z - 0.25 * math.pi))
        for nu, ph in ((0, 1.0), (1, -1j)):
            a = [1.0]
            for m in range(1, 22):
                a.append(a[-1] * (4.0 * nu * nu - (2 * m - 1) ** 2) / (8.0 * m))
            acc = torch.full_like(z, a[-1])
            for c in a[-2::-1]:
                acc = acc * w + c
            out[nu][big] = ph * amp * acc
    z = x[far] * complex(1.0, kp)
    if z.numel():
        # H_nu = sqrt(2 / (pi z)) e^{i (z - nu pi / 2 - pi / 4)} / Gamma(nu + 1/2) * integral over the real line of
        # e^{-v^2} v^{2 nu} (1 + i v^2 / (2 z))^{nu - 1/2}, by the trapezoidal rule (its error falls like e^{-2 pi d / step},
        # d > 2 the distance of the branch point)
        step, g = 0.3, 0.5j / z
        s0, s1 = torch.ones_like(z), torch.zeros_like(z)
        for m in range(1, 23):
            v2 = (step * m) ** 2
            r = torch.sqrt(1.0 + v2 * g)
            s0 += (2.0 * math.exp(-v2)) / r
            s1 += (4.0 * v2 * math.exp(-v2)) * r
        amp = torch.sqrt(2.0 / (math.pi * z)) * torch.exp(1j * (z - 0.25 * math.pi)) * (step / math.sqrt(math.pi))
        out[0][far], out[1][far] = amp * s0, -1j * amp * s1
    near = ~(far | big)
    z = x[near] * complex(1.0, kp)
    if z.numel():
        # ascending series of J0, J1, Y0, Y1 (|z| <= 5)
        q = -0.25 * z * z
        t0, t1 = torch.ones_like(z), torch.ones_like(z)
        J0, J1, S0, H = t0.clone(), t1.clone(), torch.zeros_like(z), 0.0
        S1 = (1.0 - 2.0 * np.euler_gamma) * t1
        for m in range(1, 32):
            t0, t1, H = t0 * q / (m * m), t1 * q / (m * (m + 1.0)), H + 1.0 / m
            J0, J1, S0 = J0 + t0, J1 + t1, S0 - H * t0
            S1 = S1 + (2.0 * H + 1.0 / (m + 1.0) - 2.0 * np.euler_gamma) * t1
        lz = torch.log(0.5 * z)
        J1 = 0.5 * z * J1
        Y0 = (2.0 / math.pi) * ((lz + np.euler_gamma) * J0 + S0)
        Y1 = (2.0 / math.pi) * (lz * J1 - 1.0 / z - 0.25 * z * S1)
        out[0][near], out[1][near], out[2][near], out[3][near] = J0 + 1j * Y0, J1 + 1j * Y1, J0, J1
    return out


def _log_weights(x, kind):
    """Integrals of l_p(xi) l_r(eta) log d over the unit square, l the Lagrange basis on the nodes x and d = |xi - eta|
    (kind 0), 1 - xi + eta (1: the next element), 1 + xi - eta (2: the previous one)."""
    n = 80
    v, wv = _gauss01(n)
    u, wu = v ** 5, 5.0 * v ** 4 * wv                    # graded towards 0
    A, Bq = np.meshgrid(u, v, indexing="ij")
    wa = np.outer(wu, wv)
    if kind == 0:
        # distance t = u, the smaller coordinate over the remaining 1 - t
        t, lo, w = A, (1.0 - A) * Bq, wa * (1.0 - A)
        pts = [(lo + t, lo, w, np.log(t)), (lo, lo + t, w, np.log(t))]
    else:
        # distances a, b of the two coordinates from the common node, d = a + b; triangles b < a and a < b
        pts = []
        for swap in (False, True):
            a, b = (A, A * Bq) if not swap else (A * Bq, A)
            xi, eta = (1.0 - a, b) if kind == 1 else (a, 1.0 - b)
            pts.append((xi, eta, wa * A, np.log(a + b)))

    def basis(t):
        out = np.ones((len(x),) + t.shape)
        for p in range(len(x)):
            for m in range(len(x)):
                if m != p:
                    out[p] *= (t - x[m]) / (x[p] - x[m])
        return out

    return sum(np.einsum("pij,rij,ij->pr", basis(xi), basis(eta), w * lg, optimize=True) for xi, eta, w, lg in pts)


def _operators(mesh):
    """Dense S~, D, D~, N of the mesh (complex128)."""
    N, dev, h, k, kt = mesh.N, mesh.dev, mesh.h, mesh.k, mesh.kt
    tt = kt.imag / k
    ops = [torch.zeros((N, N), dtype=torch.complex128, device=dev) for _ in range(4)]

    def hats(x, w):
        return torch.stack([w * (1.0 - x), w * x])          # [a][point]

    def scatter(e, f, blocks):
        # blocks[op][a][b]: (len(e), len(f)) values of the element pairs
        for op in range(4):
            for a in range(2):
                for b in range(2):
                    ops[op].index_put_((((e + a) % N)[:, None], ((f + b) % N)[None, :]), blocks[op][a][b], accumulate=True)

    # every pair with the regular rule, then the pairs within 8 elements again with the fine and singular rules
    x, w = (torch.tensor(v, dtype=torch.float64, device=dev) for v in _gauss01(6))
    px, py, nx, ny, _ = mesh.points(x)
    W, q = hats(x, w), 6
    step = max(1, int((1 << 23) // (N * q * q)))
    f = torch.arange(N, device=dev)
    sgn = [[1.0, -1.0], [-1.0, 1.0]]
    for e0 in range(0, N, step):
        e = torch.arange(e0, min(N, e0 + step), device=dev)
        dx = px[e][:, :, None, None] - px[None, None]
        dy = py[e][:, :, None, None] - py[None, None]
        dist = (e[:, None] - f[None, :]).abs()
        keep = (torch.minimum(dist, N - dist) > 8)
        R = torch.sqrt(dx * dx + dy * dy)
        R = torch.where(keep[:, None, :, None], R, torch.full_like(R, 30.0 / k))
        gg = (dx * nx[None, None] + dy * ny[None, None]) / R
        nd = nx[e][:, :, None, None] * nx[None, None] + ny[e][:, :, None, None] * ny[None, None]
        shape = R.shape
        Hk, Ht = _hankel((k * R).reshape(-1), 0.0), _hankel((k * R).reshape(-1), tt)
        kN, kS = 0.25j * Hk[0].reshape(shape), 0.25j * Ht[0].reshape(shape)
        kD, kDt = 0.25j * k * gg * Hk[1].reshape(shape), 0.25j * kt * gg * Ht[1].reshape(shape)
        blocks = [[[None] * 2 for _ in range(2)] for _ in range(4)]
        mask = keep.to(torch.complex128)
        Wc, wc = W.to(torch.complex128), w.to(torch.complex128)
        der = torch.einsum("p,epfr,r->ef", wc, kN, wc)
        for a in range(2):
            for b in range(2):
                for op, K in ((0, kS), (1, kD), (2, kDt), (3, nd * kN)):
                    v = torch.einsum("p,epfr,r->ef", Wc[a], K, Wc[b]) * (h * h)
                    blocks[op][a][b] = mask * (sgn[a][b] * der - k * k * v if op == 3 else v)
        scatter(e, f, blocks)
        del dx, dy, R, gg, nd, Hk, Ht, kN, kS, kD, kDt, blocks
    # near band, one offset at a time; the log-singular ones by product integration
    xn, wn = _gauss01(14)
    x, w = (torch.tensor(v, dtype=torch.float64, device=dev) for v in (xn, wn))
    px, py, nx, ny, kap = mesh.points(x)
    W = hats(x, torch.ones_like(w))
    e = torch.arange(N, device=dev)
    ww = w[:, None] * w[None, :]
    for d in range(-8, 9):
        f = (e + d) % N
        dx, dy = px[:, :, None] - px[f][:, None, :], py[:, :, None] - py[f][:, None, :]
        R = torch.sqrt(dx * dx + dy * dy)
        eye = torch.eye(len(xn), dtype=torch.bool, device=dev)[None].expand_as(R) if d == 0 else torch.zeros_like(R, dtype=torch.bool)
        R = torch.where(eye, torch.full_like(R, h), R)
        gg = (dx * nx[f][:, None, :] + dy * ny[f][:, None, :]) / R
        nd = nx[:, :, None] * nx[f][:, None, :] + ny[:, :, None] * ny[f][:, None, :]
        Hk, Ht = ([t.reshape(R.shape) for t in _hankel((k * R).reshape(-1), t0)] for t0 in (0.0, tt))
        K = [0.25j * Ht[0], 0.25j * k * gg * Hk[1], 0.25j * kt * gg * Ht[1], 0.25j * Hk[0]]
        lw = None
        if abs(d) <= 1:
            kind = 0 if d == 0 else (1 if d == 1 else 2)
            lw = torch.tensor(_log_weights(xn, kind), device=dev) + ww * math.log(h)
            dl = (x[:, None] - x[None, :]).abs() if d == 0 else (1.0 - x[:, None] + x[None, :] if d == 1 else 1.0 + x[:, None] - x[None, :])
            lg = torch.log(torch.where(dl > 0, dl, torch.ones_like(dl))) + math.log(h)
            c = -1.0 / (2.0 * math.pi)
            A = [c * Ht[2], c * k * gg * Hk[3], c * kt * gg * Ht[3], c * Hk[2]]
            K = [Kx - lg * Ax for Kx, Ax in zip(K, A)]
            if d == 0:
                def limit(z):
                    v = 0.25j + c * (np.log(complex(z) / 2.0) + np.euler_gamma)
                    return torch.full_like(K[0], complex(v))
                kd = (-kap / (4.0 * math.pi)).to(torch.complex128)[:, :, None].expand_as(R)
                lim = [limit(kt), kd, kd, limit(k)]
                K = [torch.where(eye, l, v) for l, v in zip(lim, K)]
                A = [torch.where(eye, torch.full_like(v, c if op in (0, 3) else 0.0), v) for op, v in enumerate(A)]
        for op in range(4):
            for a in range(2):
                for b in range(2):
                    phi = W[a][:, None] * W[b][None, :]
                    fac = sgn[a][b] - k * k * h * h * nd * phi if op == 3 else (h * h) * phi
                    v = (ww * fac * K[op]).sum((1, 2))
                    if lw is not None:
                        v = v + (lw * fac * A[op]).sum((1, 2))
                    ops[op].index_put_(((e + a) % N, (f + b) % N), v, accumulate=True)
    return ops


def _gram(mesh, X, inverse=False):
    m = torch.arange(mesh.N, dtype=torch.float64, device=mesh.dev)
    mu = (mesh.h * (2.0 + torch.cos(2.0 * math.pi * m / mesh.N)) / 3.0)[:, None]
    F = torch.fft.fft(X, dim=0)
    return torch.fft.ifft(F / mu if inverse else F * mu, dim=0)


def _projections(mesh, angles):
    """e / eta and h of Eq. (4) for plane waves, N x B."""
    x, w = (torch.tensor(v, dtype=torch.float64, device=mesh.dev) for v in _gauss01(14))
    px, py, nx, ny, _ = mesh.points(x)
    a = torch.tensor(angles, dtype=torch.float64, device=mesh.dev)
    e = torch.zeros((mesh.N, len(a)), dtype=torch.complex128, device=mesh.dev)
    hv = torch.zeros_like(e)
    for g in range(len(x)):
        ph = torch.exp(1j * mesh.k * (px[:, g, None] * torch.cos(a) + py[:, g, None] * torch.sin(a)))
        dn = nx[:, g, None] * torch.cos(a) + ny[:, g, None] * torch.sin(a)
        for side, lam in ((0, 1.0 - x[g]), (1, x[g])):
            c = mesh.h * w[g] * lam
            e += torch.roll(c * dn * ph, side, 0)
            hv += torch.roll(c * ph, side, 0)
    return e, hv


def _far_map(mesh, phi, j):
    x, w = (torch.tensor(v, dtype=torch.float64, device=mesh.dev) for v in _gauss01(14))
    px, py, nx, ny, _ = mesh.points(x)
    a = torch.tensor(phi, dtype=torch.float64, device=mesh.dev)
    E = torch.zeros((len(a), mesh.N), dtype=torch.complex128, device=mesh.dev)
    for g in range(len(x)):
        ph = torch.exp(-1j * mesh.k * (torch.cos(a)[:, None] * px[:, g] + torch.sin(a)[:, None] * py[:, g]))
        dn = torch.cos(a)[:, None] * nx[:, g] + torch.sin(a)[:, None] * ny[:, g]
        for side, lam in ((0, 1.0 - x[g]), (1, x[g])):
            E += torch.roll(mesh.h * w[g] * lam * dn * ph, side, 1)
    c = 1j * mesh.k * complex(math.sqrt(0.5), math.sqrt(0.5)) / math.sqrt(8.0 * math.pi * mesh.k)
    return c * (E @ j)


def _apply_c(mesh, ops, X):
    S, D, Dt, Nk = ops
    t1 = _gram(mesh, 0.5 * _gram(mesh, X) - D @ X, inverse=True)
    t2 = _gram(mesh, Nk @ X, inverse=True)
    return 0.5 * _gram(mesh, t1) + Dt @ t1 + S @ t2


def _currents(mesh, angles, adjoint_of=None):
    ops = _operators(mesh)
    C = _apply_c(mesh, ops, torch.eye(mesh.N, dtype=torch.complex128, device=mesh.dev))
    if adjoint_of is not None:
        return torch.linalg.solve(C.conj().t().contiguous(), adjoint_of)
    e, hv = _projections(mesh, angles)
    t1, t2 = _gram(mesh, hv, inverse=True), _gram(mesh, e, inverse=True)
    b = -1j * mesh.k * (ops[0] @ t2) - (0.5 * _gram(mesh, t1) + ops[2] @ t1)
    del ops
    return torch.linalg.solve(C, b)


def exact(case, seed):
    d = _inputs(case, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    kind = case["kind"]
    if kind == "batch":
        if case["n_max"] > DENSE_LIMIT:
            return None
        return [_currents(_Mesh("fourier", c, c["N"], dev), d["angles"]).cpu().numpy() for c in d["contours"]]
    mesh = _Mesh(d["family"], d["params"], case["N"], dev)
    if kind == "farfield":
        return _far_map(mesh, d["phi"], _block(case, d))
    if kind == "assemble":
        if case["N"] > 2 * DENSE_LIMIT:
            return None
        return _apply_c(mesh, _operators(mesh), _block(case, d))
    if case["N"] > DENSE_LIMIT:
        return None
    if kind == "general":
        x = _block(case, d)
        if case["adjoint"]:
            return _currents(mesh, None, adjoint_of=x)
        ops = _operators(mesh)
        return torch.linalg.solve(_apply_c(mesh, ops, torch.eye(mesh.N, dtype=torch.complex128, device=dev)), x)
    j = _currents(mesh, d["angles"])
    if kind == "gradient":   # the objective; its gradient has no closed form here
        F = _far_map(mesh, d["phi"], j)
        return [float((F.abs() ** 2).sum()), None]
    return j
