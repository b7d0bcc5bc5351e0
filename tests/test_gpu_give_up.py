"""Short wait limits, at which some waits of a tensor-core solve run out and others do not: the call returns, reports what
happened, and the handle's next solve gives the same numbers as before.  (A limit of 0 always runs out.)"""
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


# FP64 digits (several slabs, groups and units per block); FP32 parts; the FP32 pressure passes
@pytest.mark.parametrize("shape,prec,project", [((64, 66, 65), 0, False), ((130, 100, 99), 1, False), ((129, 131, 130), 1, True),
                                                ((64, 64, 64), 1, True), ((256, 64, 32), 1, True)])
def test_short_wait_limits_end_and_leave_the_handle_usable(fv, shape, prec, project):
    g = fv.Grid(*shape, stretch=1.0, Pr=0.71)
    torch.manual_seed(3)
    x = torch.randn(g.n, dtype=torch.float64, device="cuda").to(torch.float64 if prec == 0 else torch.float32)

    def solve():
        if project:
            out = x.clone()
            fv.fv_project(g, prec, out)
        else:
            out = torch.empty_like(x)
            fv.fv_diffusion_solve(g, prec, x, out)
        return out

    ref = solve()
    assert fv.fv_sync(g) == fv.FV_OK
    for limit in (0, 1, 2, 4, 8, 16, 32, 64, 256, 0):
        fv.fv_set_wait_limit(g, limit)
        solve()
        status = fv.fv_sync(g)
        assert status == fv.FV_ETIMEOUT or (limit > 0 and status == fv.FV_OK)
        fv.fv_set_wait_limit(g, -1)
        assert fv.fv_sync(g) == fv.FV_OK
        again = solve()
        assert fv.fv_sync(g) == fv.FV_OK and torch.equal(ref, again)
    g.close()
