"""Launches of few, long blocks that may start beside their predecessor's last ones: they must not pile up on the
multiprocessors that are free first.  Compared are a product's time and the sum of its kernels' times, each timed alone
between events (which keep them apart)."""
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


# blocks of the FP32 stencils; FP32 passes of long axes
@pytest.mark.parametrize("shape,nvec", [((96, 96, 96), 2), ((192, 192, 192), 1), ((32, 32, 32), 33), ((800, 16, 16), 1),
                                        ((300, 40, 40), 1), ((512, 20, 30), 1)])
def test_a_product_takes_no_longer_than_its_kernels_one_by_one(fv, shape, nvec):
    g = fv.Grid(*shape, stretch=1.5, Pr=0.71)
    q, V = torch.randn(g.n, device="cuda"), torch.randn(nvec * g.n, device="cuda")
    W = torch.empty_like(V)

    def product():
        if nvec > 1:
            fv.fv_jvp_project_batch(g, fv.FV_FP32, 1e3, -2.0, q, V, W, nvec)
        else:
            fv.fv_jvp_project(g, fv.FV_FP32, 1e3, -2.0, q, V, W)

    for _ in range(20):
        product()
    together = []
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(50):
            product()
        b.record()
        b.synchronize()
        together.append(a.elapsed_time(b) / 50)
    fv.fv_profile(g, True)
    for _ in range(20):
        product()
    alone = sum(ms for ms, _ in fv.fv_profile_read(g).values()) / 20
    fv.fv_profile(g, False)
    g.close()
    assert min(together) <= 0.9 * alone
