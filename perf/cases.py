"""Timed cases of the library's public entry points, and what they return in 64 bits.

A case is one call (or one whole solve) as a program that computes steady flows and their stability makes
it: the fused J.v + projection of a Krylov step, blocks of it, the projection alone, the diffusion solve of
the Newton preconditioner, the time step, Newton's method and the leading eigenvalues.  Sizes are those of
the repository's configurations (32^3 uniform FP64; 64^3, 100^3, 256^3 stretched with s = 1.5; blocks of 16
Krylov vectors) and of its tests (odd and unequal axes).

Inputs are made on the GPU from the seed: a base state of conduction plus a smooth divergence-free flow of
amplitude 0.05 sqrt(Gr), and rough divergence-free Krylov vectors of unit norm, both as discrete curls of
edge potentials (exactly divergence free on the staggered grid).  exact() evaluates the same discretisation
with plain torch operations in FP64 and dense 1D eigen-decompositions.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2210_08816_gb300 import fv

PR = 0.71
DEV = "cuda"


# ------------------------------------------------------------------------------------------ the cases
def listed():
    return [
        # one Chebyshev-filter step of the mixed eigen-solver at the paper's finest grid, norm left on the device
        dict(name="chebyshev_fp32_256", kind="chebyshev", prec=32, nx=256, ny=256, nz=256, stretch=1.5, Gr=2.0e8),
        # the same step in the plain FP64 form
        dict(name="chebyshev_fp64_256", kind="chebyshev", prec=64, nx=256, ny=256, nz=256, stretch=1.5, Gr=2.0e8),
        # one Krylov product of the 100^3 eigen-solve, mixed and plain form
        dict(name="jvp_project_fp32_100", kind="jvp_project", prec=32, nx=100, ny=100, nz=100, stretch=1.5, Gr=4.0e7),
        dict(name="jvp_project_fp64_100", kind="jvp_project", prec=64, nx=100, ny=100, nz=100, stretch=1.5, Gr=4.0e7),
        # one Krylov product on the grids where launches and latency count: 64^3 mixed, 32^3 plain FP64
        dict(name="jvp_project_fp32_64", kind="jvp_project", prec=32, nx=64, ny=64, nz=64, stretch=1.5, Gr=3.0e7),
        dict(name="jvp_project_fp64_32", kind="jvp_project", prec=64, nx=32, ny=32, nz=32, stretch=0.0, Gr=1.0e5),
        # a block of 16 Krylov vectors at one continuation point
        dict(name="batch16_fp32_64", kind="batch", prec=32, nx=64, ny=64, nz=64, stretch=1.5, Gr=3.0e7, nvec=16),
        # projection of a vector on a grid of odd, unequal axes
        dict(name="project_fp32_ragged", kind="project", prec=32, nx=150, ny=101, nz=67, stretch=1.5, Gr=1.0e6),
        # the diffusion inverse that preconditions every Newton and shifted solve of the mixed form
        dict(name="diffusion_fp32_64", kind="diffusion", prec=32, nx=64, ny=64, nz=64, stretch=1.5, Gr=3.0e7),
        # four steps of the time-dependent calculation with their energy and Nusselt histories
        dict(name="time_step_fp64_64", kind="time_step", prec=64, nx=64, ny=64, nz=64, stretch=1.5, Gr=1.0e7, nsteps=4),
        # a whole steady state: Newton from the perturbed conduction state, 32^3 uniform
        dict(name="newton_fp64_32", kind="newton", prec=64, nx=32, ny=32, nz=32, stretch=0.0, Gr=1.0e5),
        # a whole eigen-solve: the four leading eigenvalues about a smooth flow
        dict(name="eigen_fp64_16", kind="eigen", prec=64, nx=16, ny=16, nz=16, stretch=0.0, Gr=1.0e5),
    ]


def _size(rng, lo, hi):
    """A cell count, log-uniform in [lo, hi]: two in five multiples of 32, two in five even, the rest any."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    step = rng.choice([32, 32, 2, 2, 1]) if n >= 32 else rng.choice([2, 1])
    return max(lo, min(hi, int(round(n / step)) * step))


def draw(rng):
    """A case of the same ranges: every kind of single call, both precisions, axes equal or not."""
    kind = rng.choice(["chebyshev", "jvp_project", "jvp_project", "batch", "project", "diffusion", "time_step"])
    prec = 64 if kind == "time_step" else rng.choice([32, 32, 64])
    hi = {"batch": 128, "time_step": 100}.get(kind, 256 if prec == 32 else 160)
    n = [_size(rng, 16, hi)] * 3
    if rng.random() < 0.5:
        n = [_size(rng, 16, hi) for _ in range(3)]
    case = dict(kind=kind, prec=prec, nx=n[0], ny=n[1], nz=n[2], stretch=rng.choice([0.0, 1.0, 1.5, 1.5, 2.0]),
                Gr=float("%.3g" % math.exp(rng.uniform(math.log(1e5), math.log(2.5e8)))))
    if kind == "batch":
        case["nvec"] = rng.choice([2, 5, 8, 16])
    if kind == "time_step":
        case["nsteps"] = rng.choice([1, 2, 4])
    return case


# ------------------------------------------------------------------------------------------ grid metrics
class _Axis:
    """Faces of the tanh law (uniform for s = 0), widths, centre spacings and interpolation weights."""

    def __init__(self, n, s):
        i = np.arange(n + 1, dtype=np.float64)
        f = i / n if s == 0.0 else 0.5 * (1.0 + np.tanh(s * (2.0 * i / n - 1.0)) / np.tanh(s))
        k = n // 2
        f[n - k:] = 1.0 - f[k::-1]
        if n % 2 == 0:
            f[k] = 0.5
        f[0], f[n] = 0.0, 1.0
        self.n, self.f, self.dx = n, f, np.diff(f)
        self.xc = 0.5 * (f[:-1] + f[1:])
        self.dc = np.diff(self.xc)
        w = self.dx[:-1] + self.dx[1:]
        self.wl, self.wr = self.dx[1:] / w, self.dx[:-1] / w


def _axes(case):
    return [_Axis(case[k], case["stretch"]) for k in ("nx", "ny", "nz")]


def _sigma(case):
    """The shift of the gradient complement that the library's own solvers use by default."""
    return -0.5 / PR * sum(4.0 / float(a.dx.min()) ** 2 for a in _axes(case))


def _bc(vec, dim):
    shape = [1, 1, 1]
    shape[dim] = -1
    return torch.as_tensor(vec, dtype=torch.float64, device=DEV).reshape(shape)


def _cut(a, dim, lo, hi):
    return a.narrow(dim, lo, hi - lo)


def _diff(a, dim):
    n = a.shape[dim]
    return _cut(a, dim, 1, n) - _cut(a, dim, 0, n - 1)


def _wall(a, dim, lo=1, hi=1):
    pad = [0] * 6
    pad[2 * (2 - dim)], pad[2 * (2 - dim) + 1] = lo, hi
    return torch.nn.functional.pad(a, pad)


# ------------------------------------------------------------------------------------------ inputs
def _curl(ax, psi):
    """Divergence-free face velocities (slot 0 = wall) of edge potentials psi, zero on the wall edges."""
    nz, ny, nx = ax[2].n, ax[1].n, ax[0].n
    n = (nx, ny, nz)
    out = []
    for c in range(3):
        d, e = (c + 1) % 3, (c + 2) % 3
        # u_c = d psi_e / d x_d - d psi_d / d x_e; psi_e lives on edges along e (faces in c and d)
        dc, dd, de = 2 - c, 2 - d, 2 - e
        pe = _cut(psi[e], de, 0, n[e])
        pd = _cut(psi[d], dd, 0, n[d])
        u = _diff(pe, dd) / _bc(ax[d].dx, dd) - _diff(pd, de) / _bc(ax[e].dx, de)
        out.append(_cut(u, dc, 0, n[c]).contiguous())
    return out


def _potential(ax, g, smooth):
    """Three potentials on (n + 1)^3 points, zero on the walls: a few smooth modes, or noise at the grid scale."""
    shape = tuple(a.n + 1 for a in reversed(ax))
    xyz = [_bc(ax[2 - dim].f, dim) for dim in range(3)]
    bump = 16.0 ** 3
    for x in xyz:
        bump = bump * (x * (1.0 - x)) ** 2
    psi = []
    for _ in range(3):
        if smooth:
            p = torch.zeros(shape, dtype=torch.float64, device=DEV)
            for _ in range(3):
                r = torch.rand(7, generator=g, dtype=torch.float64, device=DEV)
                t = (r[0] - 0.5) * bump
                for dim in range(3):
                    t = t * torch.cos(math.pi * (3.0 * r[1 + dim] * xyz[dim] + r[4 + dim]))
                p += t
        else:
            p = torch.randn(shape, generator=g, dtype=torch.float64, device=DEV)
        for dim in range(3):
            p.narrow(dim, 0, 1).zero_()
            p.narrow(dim, shape[dim] - 1, 1).zero_()
        psi.append(p)
    return psi


def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) + 12345)
    return g


def _base_state(case, ax, g):
    """Conduction plus a smooth flow of amplitude 0.05 sqrt(Gr), FP64, 4N elements."""
    u = _curl(ax, _potential(ax, g, True))
    top = max(float(x.abs().max()) for x in u) or 1.0
    T = (1.0 - _bc(ax[0].xc, 2)).expand(ax[2].n, ax[1].n, ax[0].n)
    T = T + 0.05 * u[1] / top
    amp = 0.05 * math.sqrt(case["Gr"]) / top
    return torch.stack([amp * u[0], amp * u[1], amp * u[2], T]).contiguous().view(-1)


def _krylov(case, ax, g, count=1):
    """Rough divergence-free vectors of unit norm, FP64, count x 4N elements."""
    out = []
    for _ in range(count):
        u = _curl(ax, _potential(ax, g, False))
        scale = 1.0 / max(float(u[0].std()), 1e-30)
        T = torch.randn(u[0].shape, generator=g, dtype=torch.float64, device=DEV)
        v = torch.stack([scale * u[0], scale * u[1], scale * u[2], T]).view(-1)
        out.append(v / v.norm())
    return torch.cat(out)


def _inputs(case, seed):
    """The call's input tensors in its precision (a dict of 1D tensors)."""
    ax = _axes(case)
    g = _generator(seed)
    kind = case["kind"]
    dt = torch.float32 if case["prec"] == 32 else torch.float64
    if kind in ("chebyshev", "jvp_project", "batch"):
        t = {"q": _base_state(case, ax, g), "v": _krylov(case, ax, g, case.get("nvec", 1))}
        if kind == "chebyshev":
            t["w"] = _krylov(case, ax, g)
    elif kind == "project":  # what a correction step hands over: noise, not divergence free
        v = torch.randn(4, ax[2].n, ax[1].n, ax[0].n, generator=g, dtype=torch.float64, device=DEV)
        for c in range(3):
            v[c].narrow(2 - c, 0, 1).zero_()
        t = {"v": v.view(-1)}
    elif kind == "diffusion":  # a Krylov vector that Newton's preconditioner is applied to
        t = {"v": _krylov(case, ax, g)}
    elif kind == "newton":  # conduction with a perturbation of size 1e-3
        u = _curl(ax, _potential(ax, g, False))
        top = max(float(x.abs().max()) for x in u) or 1.0
        T = (1.0 - _bc(ax[0].xc, 2)).expand(ax[2].n, ax[1].n, ax[0].n).clone()
        t = {"q": torch.stack([1e-3 / top * u[0], 1e-3 / top * u[1], 1e-3 / top * u[2], T]).contiguous().view(-1)}
    else:
        t = {"q": _base_state(case, ax, g)}
    return {k: x.to(dt).contiguous() for k, x in t.items()}


def _time_dt(case):
    """A step of one tenth of the convective limit of the base state."""
    return 0.1 * min(float(a.dx.min()) for a in _axes(case)) / (0.05 * math.sqrt(case["Gr"]))


def _recurrence(case):
    """Coefficients of one step of the filter's three-term recurrence on [-2 |sigma|, 0]."""
    s = _sigma(case)
    half = 10.0 - s
    tau = 1.0 / half
    tn = 1.0 / (2.0 * half - 0.9 * s * s * tau)
    return s, 2.0 * tn, -2.0 * tn * s, -0.9 * s * s * tau * tn


# ------------------------------------------------------------------------------------------ the calls
def prepare(case, seed):
    s = dict(case=case, prec=fv.FV_FP32 if case["prec"] == 32 else fv.FV_FP64, sigma=_sigma(case))
    s["g"] = fv.Grid(case["nx"], case["ny"], case["nz"], stretch=case["stretch"], Pr=PR)
    s.update(_inputs(case, seed))
    kind = case["kind"]
    if kind in ("chebyshev", "jvp_project", "batch", "diffusion"):
        s["out"] = torch.empty_like(s["v"])
    if kind == "chebyshev":
        s["norm2"] = torch.zeros(1, dtype=torch.float64, device=DEV)
        s["coeff"] = _recurrence(case)
    if kind == "project":
        s["out"] = torch.empty_like(s["v"])
    if kind in ("time_step", "newton"):
        s["out"] = torch.empty_like(s["q"])
        s["dt"] = _time_dt(case)
    if kind == "newton":
        o = fv.fv_newton_default_opts()
        o.tol = 1e-11
        o.gr_start, o.gr_ratio = 1.25e4, 2.0
        s["opts"] = o
    if kind == "eigen":
        o = fv.fv_arnoldi_default_opts()
        o.tol, o.max_degree = 1e-10, 100
        s["opts"] = o
    return s


def run(s):
    case, g, kind = s["case"], s["g"], s["case"]["kind"]
    if kind == "chebyshev":
        sigma, alpha, beta, gamma = s["coeff"]
        fv.fv_jvp_project_lincomb_dev(g, s["prec"], case["Gr"], sigma, s["q"], s["v"], s["w"], alpha, beta, gamma,
                                      s["out"], s["norm2"])
        return [s["out"], s["norm2"]]
    if kind == "jvp_project":
        fv.fv_jvp_project(g, s["prec"], case["Gr"], s["sigma"], s["q"], s["v"], s["out"])
        return s["out"]
    if kind == "batch":
        fv.fv_jvp_project_batch(g, s["prec"], case["Gr"], s["sigma"], s["q"], s["v"], s["out"], case["nvec"],
                                use_graph=True)
        return s["out"]
    if kind == "project":
        s["out"].copy_(s["v"])
        fv.fv_project(g, s["prec"], s["out"])
        return s["out"]
    if kind == "diffusion":
        fv.fv_diffusion_solve(g, s["prec"], s["v"], s["out"])
        return s["out"]
    if kind == "time_step":
        s["out"].copy_(s["q"])
        ekin, nu = fv.fv_time_step(g, case["Gr"], s["dt"], case["nsteps"], s["out"])
        return [s["out"], np.array(ekin), np.array(nu)]
    if kind == "newton":
        s["out"].copy_(s["q"])
        st, _ = fv.newton_steady(g, case["Gr"], s["out"], s["opts"])
        return [s["out"], st]
    st, lam, _ = fv.arnoldi_leading(g, 4, case["Gr"], s["q"], s["opts"])
    return [np.array([z.real for z in lam]), np.array([abs(z.imag) for z in lam]), st]


def work(case):
    """Bytes: each input and output once.  Flops: the stencil's terms (about 300 per cell for the four
    equations of J.v, 200 for F) and, per pressure or diffusion solve, six contractions of an axis of n cells
    with the two half-size matrices that a mirror-symmetric axis needs (n flops per cell and axis)."""
    N = case["nx"] * case["ny"] * case["nz"]
    e = 4 if case["prec"] == 32 else 8
    solve = 2.0 * N * (case["nx"] + case["ny"] + case["nz"])
    jvp = 300.0 * N + solve + 30.0 * N
    kind, nv = case["kind"], case.get("nvec", 1)
    if kind == "chebyshev":
        return {"bytes": 16 * N * e, "flops": jvp}
    if kind in ("jvp_project", "batch"):
        return {"bytes": (4 + 8 * nv) * N * e, "flops": nv * jvp}
    if kind == "project":
        return {"bytes": 6 * N * e, "flops": solve + 30.0 * N}
    if kind == "diffusion":
        return {"bytes": 8 * N * e, "flops": 4 * solve}
    if kind == "time_step":
        return {"bytes": 8 * N * e, "flops": case["nsteps"] * (5 * solve + 250.0 * N)}
    # whole solves: the products they cannot do without are not known beforehand; a Newton or eigen-solve of
    # these sizes takes on the order of 100 or 1000 of them
    times = 100.0 if kind == "newton" else 1000.0
    return {"bytes": 8 * N * e, "flops": times * jvp}


# ------------------------------------------------------------------------------------------ 64-bit values
class _Exact:
    """The discretisation in plain torch FP64: face arrays with both walls, dense 1D decompositions."""

    def __init__(self, case):
        self.ax = _axes(case)
        self.n = [a.n for a in self.ax]
        self.Gr = case["Gr"]

    def full(self, x):
        x = x.double().view(4, self.n[2], self.n[1], self.n[0])
        out = [_wall(_cut(x[c], 2 - c, 1, self.n[c]), 2 - c) for c in range(3)]
        return out + [x[3].clone()]

    def flat(self, q):
        out = []
        for c in range(3):
            out.append(_cut(q[c], 2 - c, 0, self.n[c]))
        return torch.stack(out + [q[3]]).reshape(-1)

    def to_faces(self, a, d):
        """Linear interpolation of cell values to the interior faces of axis d."""
        n, dim = self.n[d], 2 - d
        return _bc(self.ax[d].wl, dim) * _cut(a, dim, 0, n - 1) + _bc(self.ax[d].wr, dim) * _cut(a, dim, 1, n)

    def convect(self, a, b):
        """div(a b) of the face velocities a and the state b, on interior faces and cells."""
        out = []
        for c in range(3):
            cd, acc = 2 - c, 0.0
            for d in range(3):
                dim = 2 - d
                if d == c:
                    mid = [0.5 * (_cut(x[c], cd, 0, self.n[c]) + _cut(x[c], cd, 1, self.n[c] + 1)) for x in (a, b)]
                    acc = acc + _diff(mid[0] * mid[1], cd) / _bc(self.ax[c].dc, cd)
                else:
                    ad = self.to_faces(a[d], c)
                    bd = _wall(self.to_faces(_cut(b[c], cd, 1, self.n[c]), d), dim)
                    acc = acc + _diff(ad * bd, dim) / _bc(self.ax[d].dx, dim)
            out.append(acc)
        acc = 0.0
        for d in range(3):
            dim = 2 - d
            acc = acc + _diff(a[d] * _wall(self.to_faces(b[3], d), dim), dim) / _bc(self.ax[d].dx, dim)
        return out + [acc]

    def spread(self, a, d, wall_lo, wall_hi):
        """d/dx (d a / dx) of cell values along axis d; wall values given (None: zero flux)."""
        dim, x = 2 - d, self.ax[d]
        n = x.n
        lo, hi = _cut(a, dim, 0, 1), _cut(a, dim, n - 1, n)
        glo = torch.zeros_like(lo) if wall_lo is None else (lo - wall_lo) * (2.0 / x.dx[0])
        ghi = torch.zeros_like(hi) if wall_hi is None else (wall_hi - hi) * (2.0 / x.dx[-1])
        g = torch.cat([glo, _diff(a, dim) / _bc(x.dc, dim), ghi], dim)
        return _diff(g, dim) / _bc(x.dx, dim)

    def laplace(self, b, hot):
        out = []
        for c in range(3):
            cd, acc = 2 - c, 0.0
            inner = _cut(b[c], cd, 1, self.n[c])
            for d in range(3):
                if d == c:
                    acc = acc + _diff(_diff(b[c], cd) / _bc(self.ax[c].dx, cd), cd) / _bc(self.ax[c].dc, cd)
                else:
                    acc = acc + self.spread(inner, d, 0.0, 0.0)
            out.append(acc)
        T = self.spread(b[3], 0, hot, 0.0) + self.spread(b[3], 1, None, None) + self.spread(b[3], 2, None, None)
        return out + [T / PR]

    def finish(self, conv, lap, T):
        r = [lap[c] - conv[c] for c in range(4)]
        r[2] = r[2] + self.Gr * self.to_faces(T, 2)
        return [_wall(r[c], 2 - c) for c in range(3)] + [r[3]]

    def jvp(self, q, v):
        ab, ba = self.convect(q, v), self.convect(v, q)
        return self.finish([ab[c] + ba[c] for c in range(4)], self.laplace(v, 0.0), v[3])

    def residual(self, q):
        return self.finish(self.convect(q, q), self.laplace(q, 1.0), q[3])

    @staticmethod
    def modes(K, w):
        """lam, E, E^-1 of the operator K that is symmetric in the weights w."""
        r = np.sqrt(w)
        S = K * r[:, None] / r[None, :]
        lam, Y = np.linalg.eigh(0.5 * (S + S.T))
        t = lambda x: torch.as_tensor(np.ascontiguousarray(x), device=DEV)  # noqa: E731
        return t(lam), t(Y / r[:, None]), t(Y.T * r[None, :])

    def cell_operator(self, d, dirichlet):
        x = self.ax[d]
        n = x.n
        G = np.zeros((n + 1, n))
        for f in range(1, n):
            G[f, f], G[f, f - 1] = 1.0 / x.dc[f - 1], -1.0 / x.dc[f - 1]
        if dirichlet:
            G[0, 0], G[n, n - 1] = 2.0 / x.dx[0], -2.0 / x.dx[-1]
        return self.modes((G[1:] - G[:-1]) / x.dx[:, None], x.dx)

    def face_operator(self, d):
        x = self.ax[d]
        n = x.n
        G = np.zeros((n, n - 1))
        for c in range(n):
            if c < n - 1:
                G[c, c] = 1.0 / x.dx[c]
            if c > 0:
                G[c, c - 1] = -1.0 / x.dx[c]
        return self.modes((G[1:] - G[:-1]) / x.dc[:, None], x.dc)

    @staticmethod
    def solve(ops, b, scale=1.0, shift=0.0, null=False):
        """(scale * (sum of the three 1D operators) - shift)^-1 b; null: the constant mode is left out."""
        L = 0.0
        for d in range(3):
            lam, _, Ei = ops[d]
            b = torch.movedim(torch.tensordot(Ei, b, ([1], [2 - d])), 0, 2 - d)
            shape = [1, 1, 1]
            shape[2 - d] = -1
            L = L + lam.reshape(shape)
        L = scale * L - shift
        if null:
            at = torch.argmin(L.abs())
            L.view(-1)[at] = 1.0
            b = b / L
            b.view(-1)[at] = 0.0
        else:
            b = b / L
        for d in range(3):
            b = torch.movedim(torch.tensordot(ops[d][1], b, ([1], [2 - d])), 0, 2 - d)
        return b

    def project(self, q):
        if not hasattr(self, "neumann"):
            self.neumann = [self.cell_operator(d, False) for d in range(3)]
        div = sum(_diff(q[d], 2 - d) / _bc(self.ax[d].dx, 2 - d) for d in range(3))
        phi = self.solve(self.neumann, div, null=True)
        return [q[d] - _wall(_diff(phi, 2 - d) / _bc(self.ax[d].dc, 2 - d), 2 - d) for d in range(3)] + [q[3]]

    def diffuse(self, q, shift=0.0):
        """(L - shift)^-1 q, field by field."""
        if not hasattr(self, "dirichlet"):
            self.dirichlet = [self.cell_operator(d, True) for d in range(3)]
            self.neumann = [self.cell_operator(d, False) for d in range(3)]
            self.face = [self.face_operator(d) for d in range(3)]
        out = []
        for c in range(3):
            ops = [self.face[d] if d == c else self.dirichlet[d] for d in range(3)]
            out.append(_wall(self.solve(ops, _cut(q[c], 2 - c, 1, self.n[c]), 1.0, shift), 2 - c))
        ops = [self.dirichlet[0], self.neumann[1], self.neumann[2]]
        return out + [self.solve(ops, q[3], 1.0 / PR, shift)]

    def energy(self, q):
        e = 0.0
        for c in range(3):
            vol = 1.0
            for d in range(3):
                w = np.concatenate([[0.0], self.ax[d].dc, [0.0]]) if d == c else self.ax[d].dx
                vol = vol * _bc(w, 2 - d)
            e = e + 0.5 * float((q[c] ** 2 * vol).sum())
        return e

    def nusselt(self, q):
        a = _bc(self.ax[1].dx, 1)[:, :, 0] * _bc(self.ax[2].dx, 0)[:, :, 0]
        return float(((q[3][:, :, 0] - 1.0) * (2.0 / self.ax[0].dx[0]) * a).sum())


def exact(case, seed):
    kind = case["kind"]
    if kind in ("newton", "eigen"):
        return None
    t = _inputs(case, seed)
    E = _Exact(case)
    if kind == "project":
        return E.flat(E.project(E.full(t["v"])))
    if kind == "diffusion":
        return E.flat(E.diffuse(E.full(t["v"])))
    if kind == "time_step":
        dt = _time_dt(case)
        q = E.full(t["q"])
        ekin, nu = [E.energy(q)], [E.nusselt(q)]
        for _ in range(case["nsteps"]):
            # q + P (1 - dt L)^-1 dt F(q)
            step = E.project(E.diffuse(E.residual(q), 1.0 / dt))
            q = [a - b for a, b in zip(q, step)]
            ekin.append(E.energy(q))
            nu.append(E.nusselt(q))
        return [E.flat(q), np.array(ekin), np.array(nu)]
    q = E.full(t["q"])
    if kind == "chebyshev":
        s, alpha, beta, gamma = _recurrence(case)
        v = E.full(t["v"])
        # alpha (P (J v - s v) + s v) + beta v + gamma w
        r = E.project([a - s * b for a, b in zip(E.jvp(q, v), v)])
        out = E.flat([alpha * (a + s * b) + beta * b for a, b in zip(r, v)]) + gamma * t["w"].double()
        return [out, (out * out).sum().reshape(1)]
    s = _sigma(case)
    outs = []
    for v in t["v"].view(case.get("nvec", 1), -1):
        v = E.full(v)
        r = E.project([a - s * b for a, b in zip(E.jvp(q, v), v)])
        outs.append(E.flat([a + s * b for a, b in zip(r, v)]))
    return torch.cat(outs)
