"""The FP64 stencils (flux form) at the sizes where their tiles can go wrong: the smallest axes, widths around the
32-cell tile and its even splits, odd rows (the form without TMA), chunks of one plane and many; F, J.v with a shift and
blocks of vectors, against the oracle.  Tolerance 1e-12 of each field's largest value, as the parity tests: a few dozen
roundings of terms of the result's own size (rough seeded data)."""
import numpy as np
import pytest

import oracle.discretisation as D
from paper_2210_08816_gb300 import seeded

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
PR = 0.71
SIZES = [(2, 3, 5), (3, 2, 2), (31, 8, 40), (32, 33, 3), (33, 17, 9), (34, 5, 70), (64, 48, 34), (70, 3, 2), (100, 21, 6),
         (126, 19, 33), (130, 12, 7)]


@pytest.fixture(scope="module")
def fv():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2210_08816_gb300 import build
    build.build()
    from paper_2210_08816_gb300 import fv as _fv
    _fv.lib()
    return _fv


def _close(got, ref, what):
    for c in range(4):
        assert np.max(np.abs(got[c] - ref[c])) <= 1e-12 * max(np.max(np.abs(ref[c])), 1e-300), f"{what}: field {c}"


@pytest.mark.parametrize("shape", SIZES)
def test_flux_stencils_match_oracle(fv, shape):
    stretch, Gr = (1.5 if sum(shape) % 2 else 0.0), 3.0e3
    og = D.Grid(*shape, stretch=stretch, Pr=PR)
    g = fv.Grid(*shape, stretch=stretch, Pr=PR)
    raw = seeded.normal_fields(31, og.shape)
    qf, v1, v2 = D.from_api(og, raw), *(D.from_api(og, seeded.normal_fields(s, og.shape)) for s in (32, 33))
    dev = lambda a: torch.tensor(np.stack(a), dtype=torch.float64, device="cuda").contiguous().view(-1)  # noqa: E731
    host = lambda t: t.view(4, *og.shape).cpu().numpy()  # noqa: E731
    # F ignores what the wall slots hold: `raw` still has its numbers there
    out = torch.empty(g.n, dtype=torch.float64, device="cuda")
    fv.fv_residual(g, Gr, dev(raw), out)
    _close(host(out), D.to_api(og, D.residual_full(og, Gr, qf)), "F")
    q, a, b = (dev(D.to_api(og, x)) for x in (qf, v1, v2))
    fv.fv_jvp(g, fv.FV_FP64, Gr, q, a, out)
    _close(host(out), D.to_api(og, D.jvp_full(og, Gr, qf, v1)), "J.v")
    # odd base address: the form without TMA gives the same numbers
    shifted = torch.empty(g.n + 1, dtype=torch.float64, device="cuda")[1:]
    shifted.copy_(a)
    again = torch.empty_like(out)
    fv.fv_jvp(g, fv.FV_FP64, Gr, q, shifted, again)
    assert torch.equal(out, again)
    # blocks with the shift against single vectors
    W, one = torch.empty(2 * g.n, dtype=torch.float64, device="cuda"), torch.empty_like(out)
    fv.fv_jvp_project_batch(g, fv.FV_FP64, Gr, -7.0, q, torch.cat([a, b]), W, 2)
    for k, x in enumerate((a, b)):
        fv.fv_jvp_project(g, fv.FV_FP64, Gr, -7.0, q, x, one)
        assert float((W[k * g.n:(k + 1) * g.n] - one).norm()) <= 1e-13 * float(one.norm())
    assert fv.fv_sync(g) == fv.FV_OK
    g.close()
