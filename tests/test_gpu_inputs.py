"""Inputs at the ends of what the FP32 tensor-core passes scale, and faces that are mirror-symmetric only to round-off."""
import numpy as np
import pytest

import oracle.discretisation as D

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
# axes of a multiple of 32 (FP16 parts under one scale per field); others (a scale per row); the CUDA cores
SHAPES = [(64, 64, 64), (96, 32, 64), (100, 90, 101), (30, 31, 32)]


@pytest.fixture(scope="module")
def fv():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2210_08816_gb300 import build
    build.build()
    from paper_2210_08816_gb300 import fv as _fv
    _fv.lib()
    return _fv


def _state(g, seed):
    torch.manual_seed(seed)
    nz, ny, nx = g.shape
    x = torch.randn(4, nz, ny, nx, device="cuda")
    x[0, :, :, 0] = x[1, :, 0] = x[2, 0] = 0.0
    return x


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_fp32_solves_keep_non_finite_inputs_visible(fv, shape, bad):
    g = fv.Grid(*shape, stretch=1.5, Pr=0.71)
    x = _state(g, 1)
    v = x.clone()
    v[0, 3, 4, 5] = bad
    fv.fv_project(g, fv.FV_FP32, v.view(-1))
    inner = v[0, :, :, 1:], v[1, :, 1:], v[2, 1:]
    assert not any(bool(torch.isfinite(f).any()) for f in inner) and torch.equal(v[3], x[3])
    b = x.clone()
    b[3, 2, 1, 7] = bad
    out = torch.zeros_like(b)
    fv.fv_diffusion_solve(g, fv.FV_FP32, b.view(-1), out.view(-1))
    assert not bool(torch.isfinite(out[3]).any()) and bool(torch.isfinite(out[:3]).all())
    # and the next solve is not affected: the fields' maxima start from zero
    w, ref = x.clone(), x.clone()
    fv.fv_project(g, fv.FV_FP32, w.view(-1))
    h = fv.Grid(*shape, stretch=1.5, Pr=0.71)
    fv.fv_project(h, fv.FV_FP32, ref.view(-1))
    assert torch.equal(w, ref)
    g.close()
    h.close()


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("power", [-60, -30, 30, 60])
def test_fp32_projection_commutes_with_powers_of_two(fv, shape, power):
    """Scaling by a power of two is exact everywhere, so the results are the same bits, scaled."""
    g = fv.Grid(*shape, stretch=1.5, Pr=0.71)
    a = _state(g, 2)
    b = a * 2.0 ** power
    fv.fv_project(g, fv.FV_FP32, a.view(-1))
    fv.fv_project(g, fv.FV_FP32, b.view(-1))
    assert torch.equal(a * 2.0 ** power, b)
    z = torch.zeros_like(a)
    fv.fv_project(g, fv.FV_FP32, z.view(-1))
    assert not bool(z.any())
    g.close()


@pytest.mark.parametrize("shape", [(64, 65, 66), (40, 33, 48)])
def test_faces_symmetric_to_round_off(fv, shape):
    """Faces moved by up to four units of round-off still take the half-size operators, made from the mean of the axis' two
    halves.  The divergence left over is what the faces' rounding makes of it: the relative change of the narrowest width,
    times the sums' own sqrt(6 n) roundings."""
    rng = np.random.default_rng(4)
    faces = []
    for n in shape:
        f = D.Axis(n, 1.5).xf.copy()
        f[1:-1] += rng.integers(-2, 3, n - 1) * 2.0 ** -53
        faces.append(f)
    g = fv.Grid(*shape, Pr=0.71, faces=faces)
    x = _state(g, 3).double()
    _, left = fv.fv_project(g, fv.FV_FP64, x.view(-1), max_it=1, want_div=True)
    narrow = min(float(np.diff(f).min()) for f in faces)
    assert left <= np.sqrt(6.0 * max(shape)) * 4.0 * 2.0 ** -53 / narrow
    g.close()
