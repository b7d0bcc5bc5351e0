"""E_kin and Nu on grids of short, long, odd and few rows against NumPy sums, and the kernels' time on short rows.

Tolerance: sums of at most 3 N positive terms (E_kin) and ny nz fluxes, of a few roundings each, added in chunks: 64 eps of
the sum of magnitudes."""
import numpy as np
import pytest

import oracle.discretisation as D

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


@pytest.mark.parametrize("shape", [(2, 3, 5), (2, 130, 131), (16, 16, 300), (31, 33, 7), (33, 2, 2), (300, 9, 8), (64, 64, 64)])
def test_sums_match_numpy(fv, shape):
    og = D.Grid(*shape, stretch=1.5, Pr=0.71)
    g = fv.Grid(*shape, Pr=0.71, faces=[a.xf for a in og.axes])
    q = np.random.default_rng(5).standard_normal((4, *og.shape))
    q[0, :, :, 0] = q[1, :, 0, :] = q[2, 0] = 0.0
    ekin, nu = fv.fv_diagnostics(g, torch.tensor(q, device="cuda").view(-1))
    g.close()
    dx = [a.dx for a in og.axes]
    spacing = [np.concatenate([[d[0] / 2], (d[1:] + d[:-1]) / 2]) for d in dx]
    want = 0.0
    for c in range(3):
        w = [spacing[d] if d == c else dx[d] for d in range(3)]
        want += 0.5 * np.sum(q[c] ** 2 * w[2][:, None, None] * w[1][None, :, None] * w[0][None, None, :])
    flux = (q[3, :, :, 0] - 1.0) * 2.0 / dx[0][0] * dx[2][:, None] * dx[1][None, :]
    eps = 64 * np.finfo(np.float64).eps
    assert abs(ekin - want) <= eps * want
    assert abs(abs(nu) - abs(flux.sum())) <= eps * np.abs(flux).sum()


def test_short_rows_take_no_longer_than_long_ones(fv):
    """The same number of cells in rows of 16 and of 800: the factor of a row must not cost more than the row."""
    def kernels(shape):
        g = fv.Grid(*shape, stretch=1.0, Pr=0.71)
        q = torch.randn(g.n, dtype=torch.float64, device="cuda")
        for _ in range(3):
            fv.fv_diagnostics(g, q)
        fv.fv_profile(g, True)
        for _ in range(20):
            fv.fv_diagnostics(g, q)
        ms = fv.fv_profile_read(g)["reduce"][0]
        fv.fv_profile(g, False)
        g.close()
        return ms
    assert kernels((16, 16, 800)) <= 1.5 * kernels((800, 16, 16))
