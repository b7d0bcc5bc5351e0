"""The projection on strongly stretched grids, where the widths of an axis span a factor of hundreds to tens of thousands.

Reference: the same faces, solved by NumPy decompositions and refined with residuals in extended precision.  Compared is
the correction G phi, field by field.  It divides differences of neighbouring potentials by the narrowest widths, so one
rounding of the potential (eps) shows as eps times the ratio of the widest to the narrowest.  FP64: the six transforms and
the decompositions make ~6 n roundings that add at random, sqrt(6 n) eps ratio.  FP32: the decompositions are rounded from
FP64 and the sums are half as long; the six stored fields' roundings count, sqrt(6) eps ratio, twice that allowed."""
import numpy as np
import pytest

import oracle.discretisation as D

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
LD = np.longdouble


@pytest.fixture(scope="module")
def fv():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2210_08816_gb300 import build
    build.build()
    from paper_2210_08816_gb300 import fv as _fv
    _fv.lib()
    return _fv


def _along(v, axis):
    return v.reshape([-1 if a == axis else 1 for a in range(3)])


def _gradient_of_potential(og, f):
    """G phi with D G phi = D f, arrays (z, y, x) of the interior faces, in extended precision."""
    dx = [np.diff(a.xf.astype(LD)) for a in og.axes]
    dc = [(d[1:] + d[:-1]) / 2 for d in dx]
    modes = []
    for d, c in zip(dx, dc):
        n = len(d)
        L = np.zeros((n, n))
        for i in range(n - 1):
            s = float(1 / (c[i] * np.sqrt(d[i] * d[i + 1])))
            L[i, i] -= float(1 / (c[i] * d[i]))
            L[i + 1, i + 1] -= float(1 / (c[i] * d[i + 1]))
            L[i, i + 1] = L[i + 1, i] = s
        lam, Y = np.linalg.eigh(L)
        modes.append((lam, Y, np.sqrt(d.astype(np.float64))))

    def apply(M, b, d):
        return np.moveaxis(np.tensordot(M, b, ([1], [2 - d])), 0, 2 - d)

    def solve(r):
        b, L = r.astype(np.float64), 0.0
        for d, (lam, Y, w) in enumerate(modes):
            b = apply(Y.T * w, b, d)
            L = L + _along(lam, 2 - d)
        at = np.unravel_index(np.argmax(L), L.shape)
        L[at] = 1.0
        b = b / L
        b[at] = 0.0
        for d, (lam, Y, w) in enumerate(modes):
            b = apply(Y / w[:, None], b, d)
        return b

    def grad(phi):
        return [np.diff(phi, axis=2 - d) / _along(dc[d], 2 - d) for d in range(3)]

    def div(g):
        pad = [[(1, 1) if a == 2 - d else (0, 0) for a in range(3)] for d in range(3)]
        return sum(np.diff(np.pad(g[d], pad[d]), axis=2 - d) / _along(dx[d], 2 - d) for d in range(3))

    rhs = div([f[d].astype(LD) for d in range(3)])
    W = _along(dx[0], 2) * _along(dx[1], 1) * _along(dx[2], 0)
    phi = np.zeros_like(rhs)
    for _ in range(4):
        r = rhs - div(grad(phi))
        phi = phi + solve(r - (r * W).sum() / W.sum())
    return grad(phi)


def _check_projection(fv, shape, stretch, prec, factor):
    og = D.Grid(*shape, stretch=stretch, Pr=0.71)
    g = fv.Grid(*shape, Pr=0.71, faces=[a.xf for a in og.axes])
    dt = torch.float64 if prec == 0 else torch.float32
    rng = np.random.default_rng(11)
    v = rng.standard_normal((4, *og.shape)).astype(np.float64 if prec == 0 else np.float32).astype(np.float64)
    v[0, :, :, 0] = v[1, :, 0, :] = v[2, 0] = 0.0
    x = torch.tensor(v, dtype=dt, device="cuda").view(-1)
    fv.fv_project(g, prec, x)
    assert fv.fv_sync(g) == fv.FV_OK
    got = v - x.view(4, *og.shape).double().cpu().numpy()
    g.close()
    inner = [D._sl(2 - d, slice(1, None)) for d in range(3)]
    ref = _gradient_of_potential(og, [v[d][inner[d]] for d in range(3)])
    ratio = max(float(np.max(a.dx) / np.min(a.dx)) for a in og.axes)
    for d in range(3):
        e = got[d][inner[d]] - ref[d]
        rel = float(np.sqrt((e ** 2).sum() / (ref[d] ** 2).sum()))
        assert rel <= factor * (2.0 ** -53 if prec == 0 else 2.0 ** -24) * ratio, f"field {d}: {rel:.2e}, ratio {ratio:.0f}"


@pytest.mark.parametrize("shape", [(128, 40, 36), (64, 66, 65), (49, 100, 130)])
@pytest.mark.parametrize("stretch", [4.0, 6.0])
def test_fp64_projection_keeps_its_accuracy(fv, shape, stretch):
    _check_projection(fv, shape, stretch, 0, np.sqrt(6.0 * max(shape)))


# multiples of 32: by FP16 parts under one scale per field while the widths allow it
@pytest.mark.parametrize("shape", [(128, 64, 32), (64, 64, 64), (130, 70, 60), (30, 41, 36)])
@pytest.mark.parametrize("stretch", [2.0, 4.0, 4.2, 6.0])
def test_fp32_projection_keeps_its_accuracy(fv, shape, stretch):
    _check_projection(fv, shape, stretch, 1, 2.0 * np.sqrt(6.0))
