"""The half-size 1D operators of a mirror-symmetric axis (csrc/host_grid.cpp, build_half_op) on the CPU: folded out
to full size they are inverse pairs of transforms that diagonalise the dense operators of build_axis."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
DP = np.ctypeslib.ndpointer(dtype=np.float64, flags="C_CONTIGUOUS")

WRAP = r"""
#include <cstring>
#include "fv_internal.h"
namespace fv { void set_error(const std::string&) {} }
extern "C" int half_op(int n, double s, int kind, int* k0S, double* lam, double* F0, double* F1, double* E0, double* E1,
                       double* dlam, double* dEinv, double* dE, double* W) {
  fv::AxisHost a;
  if (fv::build_axis(fv::tanh_faces(n, s), a) != FV_OK) return -1;
  fv::HalfOpHost o;
  if (fv::build_half_op(a, kind, o) != FV_OK) return -2;
  k0S[0] = o.k0; k0S[1] = o.S;
  auto put = [](double* d, const std::vector<double>& v) { std::memcpy(d, v.data(), sizeof(double) * v.size()); };
  put(lam, o.lam); put(F0, o.F[0]); put(F1, o.F[1]); put(E0, o.E[0]); put(E1, o.E[1]);
  put(dlam, kind == 0 ? a.lam : kind == 1 ? a.cd_lam : a.fd_lam);
  put(dEinv, kind == 0 ? a.Einv : kind == 1 ? a.cd_Einv : a.fd_Einv);
  put(dE, kind == 0 ? a.E : kind == 1 ? a.cd_E : a.fd_E);
  for (int i = 0; i < n; ++i) W[i] = kind == 2 ? 1.0 / a.idc[i] : 1.0 / a.idx[i];
  return 0;
}
"""


@pytest.fixture(scope="module")
def half_op(tmp_path_factory):
    d = tmp_path_factory.mktemp("half")
    src, out = d / "wrap.cpp", d / "libhalf.so"
    src.write_text(WRAP)
    csrc = os.path.join(ROOT, "paper_2210_08816_gb300", "csrc")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f"-I{cuda}/include", f"-I{csrc}", str(src),
                        os.path.join(csrc, "host_grid.cpp"), os.path.join(csrc, "host_linalg.cpp"), "-o", str(out)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    f = C.CDLL(str(out)).half_op
    f.restype = C.c_int
    f.argtypes = [C.c_int, C.c_double, C.c_int, C.POINTER(C.c_int)] + [DP] * 9
    return f


@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("n,s", [(2, 0.0), (3, 1.5), (4, 0.0), (5, 2.0), (16, 1.5), (31, 0.0), (64, 1.5), (67, 2.0)])
def test_half_operator_folds_out_to_the_dense_one(half_op, n, s, kind):
    h, ha = (n + 1) // 2, n // 2
    k0S = (C.c_int * 2)()
    lam, dlam, W = np.zeros(n), np.zeros(n), np.zeros(n)
    F0, F1, E0, E1 = (np.zeros((h, h)) for _ in range(4))
    dEinv, dE = np.zeros((n, n)), np.zeros((n, n))
    assert half_op(n, s, kind, k0S, lam, F0, F1, E0, E1, dlam, dEinv, dE, W) == 0
    k0, S = k0S[0], k0S[1]
    Fw, Bw = np.zeros((n, n)), np.zeros((n, n))
    for i in range(h):           # forward: sums and differences of the pairs
        i1, i2 = k0 + i, S - k0 - i
        Fw[:h, i1] += F0[:, i]
        Fw[:h, i2] += F0[:, i]
        Fw[h:, i1] += F1[:ha, i]
        Fw[h:, i2] -= F1[:ha, i]
        if i1 <= i2:             # backward
            Bw[i1, :h] = E0[i, :]
            Bw[i1, h:] = E1[i, :ha]
            if i2 != i1:
                Bw[i2, :h] = E0[i, :]
                Bw[i2, h:] = -E1[i, :ha]
    live = np.arange(k0, n)
    A = (dE * dlam) @ dEinv      # the dense operator
    B = (Bw * lam) @ Fw
    # eigen-decompositions to n eps; the halves' mean differs from either by the faces' round-off, eps / width
    tol = (20.0 * n + 4.0 / W.min()) * np.finfo(float).eps
    r = np.sqrt(W)
    sym = lambda M: r[live, None] * M[np.ix_(live, live)] / r[None, live]  # noqa: E731  (the symmetric form)
    assert np.max(np.abs(sym(B) - sym(A))) <= tol * np.max(np.abs(sym(A)))
    assert np.max(np.abs(sym(Bw @ Fw) - np.eye(len(live)))) <= tol
    if k0:
        assert not Bw[0].any() and not Fw[:, 0].any()
    used = [m for m in range(n) if Fw[m].any()]
    assert len(used) == n - k0 and np.allclose(np.sort(lam[used]), np.sort(dlam[live]), rtol=tol, atol=tol * np.abs(dlam).max())
    if kind == 0:
        assert lam[0] == 0.0
