"""The direct solves (pressure projection, diffusion inverse) at the sizes where a pass can go wrong: the smallest
axes, odd and even ones, tile edges and remainders (31, 33, 63, 65, 129, ...), unequal axes, blocks of vectors;
against a plain NumPy FP64 solve by dense 1D eigen-decompositions of the oracle's metrics.

Tolerances, FP64: six transforms of ~n roundings each, 40 n eps.  The projection amplifies them by the difference
of neighbouring potentials over a spacing (the cell count at most): 40 n^2 eps of each field's 2-norm.  The
diffusion inverse is held to its backward error: ||L x - b|| <= 40 n eps (||L|| ||x|| + ||b||) field by field (its
forward error carries the condition number lam_max / lam_min ~ n^2 as well, in the reference's own decompositions
too).  FP32: 5e-5 of the largest value, as the projection's parity tests use."""
import numpy as np
import pytest

import oracle.discretisation as D
from paper_2210_08816_gb300 import seeded

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
PR = 0.71
SIZES = [(2, 3, 5), (4, 2, 3), (16, 16, 16), (31, 33, 32), (64, 65, 31), (100, 63, 36), (129, 40, 50), (17, 130, 66),
         (33, 20, 255), (256, 34, 48), (255, 130, 131)]


@pytest.fixture(scope="module")
def fv():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2210_08816_gb300 import build
    build.build()
    from paper_2210_08816_gb300 import fv as _fv
    _fv.lib()
    return _fv


def _modes(K, w):
    r = np.sqrt(w)
    S = K * r[:, None] / r[None, :]
    lam, Y = np.linalg.eigh(0.5 * (S + S.T))
    return lam, Y / r[:, None], Y.T * r[None, :]


def _operator(ax, kind):
    n = ax.n
    if kind == "face":
        G = np.zeros((n, n - 1))
        for c in range(n):
            if c < n - 1:
                G[c, c] = 1.0 / ax.dx[c]
            if c > 0:
                G[c, c - 1] = -1.0 / ax.dx[c]
        return _modes((G[1:] - G[:-1]) / ax.dc[:, None], ax.dc)
    G = np.zeros((n + 1, n))
    for f in range(1, n):
        G[f, f], G[f, f - 1] = 1.0 / ax.dc[f - 1], -1.0 / ax.dc[f - 1]
    if kind == "dirichlet":
        G[0, 0], G[n, n - 1] = 2.0 / ax.dx[0], -2.0 / ax.dx[-1]
    return _modes((G[1:] - G[:-1]) / ax.dx[:, None], ax.dx)


def _solve(ops, b, scale=1.0, null=False):
    L = 0.0
    for d in range(3):
        b = np.moveaxis(np.tensordot(ops[d][2], b, ([1], [2 - d])), 0, 2 - d)
        L = L + ops[d][0].reshape([-1 if a == 2 - d else 1 for a in range(3)])
    L = scale * L
    if null:
        at = np.unravel_index(np.argmin(np.abs(L)), L.shape)
        L[at] = np.inf
    b = b / L
    for d in range(3):
        b = np.moveaxis(np.tensordot(ops[d][1], b, ([1], [2 - d])), 0, 2 - d)
    return b


def _project(og, a):
    f = D.from_api(og, a)
    ax = og.axes
    div = sum(np.diff(f[c], axis=2 - c) / D._b(ax[c].dx, 2 - c) for c in range(3))
    phi = _solve([_operator(x, "neumann") for x in ax], div, null=True)
    out = [f[c] - D._pad_walls(np.diff(phi, axis=2 - c) / D._b(ax[c].dc, 2 - c), 2 - c) for c in range(3)]
    return D.to_api(og, out + [f[3]])


def _diffuse(og, a):
    ax = og.axes
    out = []
    for c in range(3):
        ops = [_operator(ax[d], "face" if d == c else "dirichlet") for d in range(3)]
        inner = a[c][D._sl(2 - c, slice(1, None))]
        x = np.zeros(og.shape)
        x[D._sl(2 - c, slice(1, None))] = _solve(ops, inner)
        out.append(x)
    ops = [_operator(ax[0], "dirichlet"), _operator(ax[1], "neumann"), _operator(ax[2], "neumann")]
    return out + [_solve(ops, a[3], 1.0 / PR)]


def _residuals(og, x, b):
    """Per field (||L x - b||, ||L|| ||x|| + ||b||) of the diffusion operators, applied as sums of 1D matrices."""
    ax = og.axes
    out = []
    for c in range(4):
        cut = D._sl(2 - c, slice(1, None)) if c < 3 else slice(None)
        xi, bi = x[c][cut], b[c][cut]
        r, norm = -bi, 0.0
        for d in range(3):
            kind = ("face" if d == c else "dirichlet") if c < 3 else ("dirichlet" if d == 0 else "neumann")
            lam, E, Ei = _operator(ax[d], kind)
            K = (E * lam) @ Ei / (PR if c == 3 else 1.0)
            r = r + np.moveaxis(np.tensordot(K, xi, ([1], [2 - d])), 0, 2 - d)
            norm += np.max(np.abs(lam)) / (PR if c == 3 else 1.0)
        out.append((np.linalg.norm(r), norm * np.linalg.norm(xi) + np.linalg.norm(bi)))
    return out


def _fields(og, seed, dt):
    a = D.to_api(og, D.from_api(og, seeded.normal_fields(seed, og.shape)))
    return [x.astype(dt).astype(np.float64) for x in a]


def _check(got, ref, n, prec64, what):
    for c in range(4):
        r = np.linalg.norm(ref[c])
        if prec64:
            tol = 40.0 * float(n) ** 2 * np.finfo(np.float64).eps
            assert np.linalg.norm(got[c] - ref[c]) <= tol * max(r, 1e-300), f"{what}: field {c}"
        else:
            assert np.max(np.abs(got[c] - ref[c])) <= 5e-5 * max(np.max(np.abs(ref[c])), 1e-30), f"{what}: field {c}"


@pytest.mark.parametrize("shape", SIZES)
@pytest.mark.parametrize("prec", [0, 1])
def test_direct_solves_match_dense_decompositions(fv, shape, prec):
    stretch = 1.5 if sum(shape) % 2 else 0.0
    og = D.Grid(*shape, stretch=stretch, Pr=PR)
    g = fv.Grid(*shape, stretch=stretch, Pr=PR)
    dt = np.float64 if prec == 0 else np.float32
    a, b = _fields(og, 5, dt), _fields(og, 6, dt)
    dev = lambda x: torch.tensor(np.stack(x), dtype=torch.float64 if prec == 0 else torch.float32, device="cuda").view(-1)  # noqa: E731
    host = lambda t: t.view(4, *og.shape).double().cpu().numpy()  # noqa: E731
    n = max(shape)
    v = dev(a)
    fv.fv_project(g, prec, v)
    _check(host(v), _project(og, a), n, prec == 0, "project")
    x = dev(b)
    out = torch.full_like(x, float("nan"))
    fv.fv_diffusion_solve(g, prec, x, out)
    if prec == 0:
        for c, (r, size) in enumerate(_residuals(og, host(out), b)):
            assert r <= 40.0 * n * np.finfo(np.float64).eps * size, f"diffusion: field {c}"
    else:
        _check(host(out), _diffuse(og, b), n, False, "diffusion")
    fv.fv_diffusion_solve(g, prec, x, x)  # in place
    assert torch.equal(x, out)
    # a block of vectors gives the single vectors' results
    q, V = dev(_fields(og, 7, dt)), torch.cat([dev(a), dev(b), dev(_fields(og, 8, dt))])
    W, one = torch.empty_like(V), torch.empty_like(q)
    fv.fv_jvp_project_batch(g, prec, 1e3, -2.0, q, V, W, 3)
    for i in range(3):
        fv.fv_jvp_project(g, prec, 1e3, -2.0, q, V[i * g.n:(i + 1) * g.n].clone(), one)
        assert float((W[i * g.n:(i + 1) * g.n] - one).norm()) <= (1e-13 if prec == 0 else 1e-5) * float(one.norm())
    assert fv.fv_sync(g) == fv.FV_OK
    g.close()


def test_digit_pass_gives_up_and_recovers(fv):
    """With a wait limit of 0 the tensor-core passes of an FP64 solve stop and report it; the handle stays usable."""
    og = D.Grid(64, 66, 65, stretch=1.0, Pr=PR)
    g = fv.Grid(64, 66, 65, stretch=1.0, Pr=PR)
    b = _fields(og, 9, np.float64)
    x = torch.tensor(np.stack(b), dtype=torch.float64, device="cuda").view(-1)
    out, again = torch.empty_like(x), torch.empty_like(x)
    fv.fv_diffusion_solve(g, 0, x, out)
    assert fv.fv_sync(g) == fv.FV_OK
    fv.fv_set_wait_limit(g, 0)
    fv.fv_diffusion_solve(g, 0, x, again)
    assert fv.fv_sync(g) == fv.FV_ETIMEOUT
    fv.fv_set_wait_limit(g, -1)
    fv.fv_diffusion_solve(g, 0, x, again)
    assert fv.fv_sync(g) == fv.FV_OK and torch.equal(out, again)
    g.close()


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_digit_pass_keeps_non_finite_inputs_visible(fv, bad):
    og = D.Grid(64, 64, 64, stretch=1.0, Pr=PR)
    g = fv.Grid(64, 64, 64, stretch=1.0, Pr=PR)
    x = torch.tensor(np.stack(_fields(og, 9, np.float64)), dtype=torch.float64, device="cuda").view(-1)
    x[3 * og.nx ** 3 + 777] = bad
    out = torch.zeros_like(x)
    fv.fv_diffusion_solve(g, 0, x, out)
    T = out.view(4, -1)
    assert not bool(torch.isfinite(T[3]).any()) and bool(torch.isfinite(T[:3]).all())
    x.zero_()
    fv.fv_diffusion_solve(g, 0, x, out)
    assert not bool(out.any())
    g.close()
