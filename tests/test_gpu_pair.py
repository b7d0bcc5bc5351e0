"""The FP32 stencils at the edges of their tiles and z-chunks (two cells per thread: nx a multiple of 64; one cell: other
sizes), against the FP64 path, and the T that they write to a step's result themselves where nothing else can still read
what it overwrites: the same step with its result elsewhere, in w and over the end of q (where the correction writes T,
when q is no longer read) gives the same numbers and the same norm.

Tolerances: 5e-5 of the largest value against FP64, as the parity tests use; between the forms the velocity bit for bit
and T to the two roundings by which a contraction may differ, 2^-22 of its terms' largest."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SIZES = [(64, 16, 2), (64, 17, 33), (128, 31, 40), (192, 40, 7), (64, 64, 64), (36, 20, 18), (67, 33, 5), (100, 16, 31)]


@pytest.fixture(scope="module")
def fv():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2210_08816_gb300 import build
    build.build()
    from paper_2210_08816_gb300 import fv as _fv
    _fv.lib()
    return _fv


def _field(shape, seed, dtype=torch.float32):
    nx, ny, nz = shape
    a = np.random.default_rng(seed).standard_normal((4, nz, ny, nx))
    a[0, :, :, 0] = a[1, :, 0, :] = a[2, 0] = 0.0
    return torch.tensor(a, dtype=torch.float32, device="cuda").to(dtype).reshape(-1)


@pytest.mark.parametrize("shape", SIZES)
def test_stencil_against_fp64(fv, shape):
    g = fv.Grid(*shape, stretch=1.5, Pr=0.71)
    q, v = _field(shape, 1), _field(shape, 2)
    out = torch.empty_like(v)
    fv.fv_jvp(g, fv.FV_FP32, 2.0e4, q, v, out)
    ref = torch.empty_like(v, dtype=torch.float64)
    fv.fv_jvp(g, fv.FV_FP64, 2.0e4, q.double(), v.double(), ref)
    o, r = out.double().view(4, -1), ref.view(4, -1)
    assert torch.all((o - r).abs().amax(1) <= 5e-5 * r.abs().amax(1))


@pytest.mark.parametrize("shape", SIZES)
def test_step_is_the_same_wherever_its_result_goes(fv, shape):
    g = fv.Grid(*shape, stretch=1.5, Pr=0.71)
    q, v, w = _field(shape, 3), _field(shape, 4), _field(shape, 5)
    Gr, sigma, al, be, ga = 3.0e4, -250.0, 0.7, 1.3, -0.4

    def step(vv, ww, out, qq=q):
        n2 = fv.fv_jvp_project_lincomb(g, fv.FV_FP32, Gr, sigma, qq, vv, ww, al, be, ga, out, want_norm=True)
        return out.view(4, -1).clone(), n2

    a, na = step(v.clone(), w.clone(), torch.empty_like(v))
    ww = w.clone()
    b, nb = step(v.clone(), ww, ww)
    n = v.numel()
    both = torch.empty(2 * n, dtype=v.dtype, device="cuda")  # the result's first 64 values are q's last ones
    both[:n] = q
    c, nc = step(v.clone(), w.clone(), both[n - 64:2 * n - 64], both[:n])
    assert torch.equal(a, b) and na == nb
    assert torch.equal(a[:3], c[:3])
    Y = torch.empty_like(v)
    big = a[3].abs().max()
    fv.fv_jvp_project_lincomb(g, fv.FV_FP32, Gr, sigma, q, v, None, al, 0.0, 0.0, Y)
    big = torch.maximum(big, Y.view(4, -1)[3].abs().max()) + 2.0 * v.view(4, -1)[3].abs().max() + w.view(4, -1)[3].abs().max()
    assert (a[3] - c[3]).abs().max() <= 2.0 ** -22 * big
    assert abs(na - nc) <= 1e-6 * nc
