"""FP32 pressure solves on the tensor cores (FP16 heads and remainders under one scale per field): axes of one and of
several steps, whole and half slabs (32, 64, 96, 160, 224, 256 cells), and fields of very different magnitude.

The scale is a power of two and every other operation of the projection and of J.v is linear, so a field times 2^k
gives 2^k times the result, bit for bit, alone and as one vector of a block, and a zero field gives zeros.  Against the
FP64 path: 5e-5 of the largest value, as the projection's parity tests use."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fv():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2210_08816_gb300 import build
    build.build()
    from paper_2210_08816_gb300 import fv as _fv
    _fv.lib()
    return _fv


def _field(shape, seed):
    nx, ny, nz = shape
    a = np.random.default_rng(seed).standard_normal((4, nz, ny, nx))
    a[0, :, :, 0] = a[1, :, 0, :] = a[2, 0] = 0.0
    return torch.tensor(a, dtype=torch.float32, device="cuda").reshape(-1)


@pytest.mark.parametrize("shape", [(32, 32, 32), (32, 224, 256), (160, 64, 96), (256, 32, 192), (96, 160, 224)])
def test_projection_and_scaling(fv, shape):
    g = fv.Grid(*shape, stretch=1.5, Pr=0.71)
    v = _field(shape, 5)
    ref = v.double()
    fv.fv_project(g, fv.FV_FP64, ref, max_it=1)
    outs = []
    for k in (0, 40, -40):
        t = v * 2.0 ** k
        fv.fv_project(g, fv.FV_FP32, t, max_it=1)
        outs.append(t)
    r, o = ref.view(4, -1), outs[0].double().view(4, -1)
    assert torch.all((o - r).abs().amax(1) <= 5e-5 * r.abs().amax(1))
    assert torch.equal(outs[1], outs[0] * 2.0 ** 40) and torch.equal(outs[2], outs[0] * 2.0 ** -40)
    z = torch.zeros_like(v)
    fv.fv_project(g, fv.FV_FP32, z, max_it=1)
    assert torch.count_nonzero(z) == 0


@pytest.mark.parametrize("shape", [(64, 64, 64), (96, 32, 160)])
def test_block_of_unequal_vectors(fv, shape):
    g = fv.Grid(*shape, stretch=1.5, Pr=0.71)
    q, v = _field(shape, 6), _field(shape, 7)
    scales = (1.0, 2.0 ** -40, 0.0, 2.0 ** 40, 2.0 ** 7)
    V = torch.cat([v * s for s in scales])
    W = torch.empty_like(V)
    for _ in range(2):  # a second call finds the maxima of the first cleared
        fv.fv_jvp_project_batch(g, fv.FV_FP32, 1.0e5, -300.0, q, V, W, len(scales))
    W = W.view(len(scales), -1)
    for i, s in enumerate(scales):
        assert torch.equal(W[i], W[0] * s)
