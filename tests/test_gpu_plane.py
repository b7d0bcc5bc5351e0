"""The FP64 solves of small grids by pairs of passes on planes (csrc/kernels_plane.cu): the projection against a dense NumPy
solve of the same discretisation is in test_gpu_solves.py; here every shape class of the planes (one block or a cluster,
odd and even axes, rows that do not divide among the blocks, unequal strides) by the residuals of the two solves, in place
and out of place.

Tolerances: the projected field's divergence falls to six transforms' rounding, 40 n eps of the largest term of a
divergence (its largest velocity over the smallest width); two projections agree to the same relative to their largest
value; the diffusion solve in place and out of place agrees bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
EPS = 2.0 ** -52
SIZES = [(2, 3, 5), (8, 8, 8), (16, 16, 16), (17, 16, 15), (24, 24, 24), (31, 33, 32), (32, 32, 32), (36, 36, 36),
         (64, 32, 16), (16, 32, 64), (7, 64, 9), (40, 40, 40)]


@pytest.fixture(scope="module")
def fv():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2210_08816_gb300 import build
    build.build()
    from paper_2210_08816_gb300 import fv as _fv
    _fv.lib()
    return _fv


def _widths(n, s):
    f = np.array([i / n if s == 0 else 0.5 * (1 + np.tanh(s * (2 * i / n - 1)) / np.tanh(s)) for i in range(n + 1)])
    return np.diff(f)


@pytest.mark.parametrize("shape", SIZES)
def test_projection_is_divergence_free_and_idempotent(fv, shape):
    nx, ny, nz = shape
    s = 1.5
    g = fv.Grid(nx, ny, nz, stretch=s, Pr=0.71)
    a = np.random.default_rng(8).standard_normal((4, nz, ny, nx))
    a[0, :, :, 0] = a[1, :, 0, :] = a[2, 0] = 0.0
    t = torch.tensor(a.reshape(-1), device="cuda")
    fv.fv_project(g, fv.FV_FP64, t, max_it=1)
    p = t.view(4, nz, ny, nx).cpu().numpy()
    w = [_widths(n, s) for n in (nx, ny, nz)]
    d = np.diff(np.concatenate([p[0], np.zeros((nz, ny, 1))], 2), axis=2) / w[0][None, None, :]
    d += np.diff(np.concatenate([p[1], np.zeros((nz, 1, nx))], 1), axis=1) / w[1][None, :, None]
    d += np.diff(np.concatenate([p[2], np.zeros((1, ny, nx))], 0), axis=0) / w[2][:, None, None]
    n = max(shape)
    assert np.abs(d).max() <= 40 * n * EPS * np.abs(a[:3]).max() / min(x.min() for x in w)
    u = t.clone()
    fv.fv_project(g, fv.FV_FP64, u, max_it=1)
    assert (u - t).abs().max() <= 40 * n * EPS * t.abs().max()
    assert torch.equal(t.view(4, -1)[3], torch.tensor(a[3].reshape(-1), device="cuda"))


@pytest.mark.parametrize("shape", SIZES)
def test_diffusion_solve_in_place(fv, shape):
    nx, ny, nz = shape
    g = fv.Grid(nx, ny, nz, stretch=1.5, Pr=0.71)
    a = np.random.default_rng(9).standard_normal((4, nz, ny, nx))
    a[0, :, :, 0] = a[1, :, 0, :] = a[2, 0] = 0.0
    x = torch.tensor(a.reshape(-1), device="cuda")
    out = torch.empty_like(x)
    fv.fv_diffusion_solve(g, fv.FV_FP64, x, out)
    y = x.clone()
    fv.fv_diffusion_solve(g, fv.FV_FP64, y, y)
    assert torch.equal(out, y) and torch.isfinite(out).all()
    o = out.view(4, nz, ny, nx)
    assert not (o[0, :, :, 0].any() or o[1, :, 0, :].any() or o[2, 0].any())


@pytest.mark.parametrize("prec,shape,nvec", [(64, (24, 20, 36), 12), (64, (40, 40, 40), 3), (64, (16, 16, 16), 9),
                                             (64, (56, 30, 44), 4), (32, (80, 40, 30), 16), (32, (68, 60, 52), 5)])
def test_block_of_vectors_is_its_vectors_one_by_one(fv, prec, shape, nvec):
    g = fv.Grid(*shape, stretch=1.5, Pr=0.71)
    p, dt = (fv.FV_FP64, torch.float64) if prec == 64 else (fv.FV_FP32, torch.float32)
    gen = torch.Generator().manual_seed(4)
    q = torch.randn(g.n, generator=gen, dtype=torch.float64).to(dt).cuda()
    V = torch.randn(nvec * g.n, generator=gen, dtype=torch.float64).to(dt).cuda()
    W, one = torch.empty_like(V), torch.empty_like(V)
    fv.fv_jvp_project_batch(g, p, 1.0e4, -90.0, q, V, W, nvec)
    for i in range(nvec):
        fv.fv_jvp_project(g, p, 1.0e4, -90.0, q, V[i * g.n:(i + 1) * g.n], one[i * g.n:(i + 1) * g.n])
    assert torch.equal(W, one)
