"""The operands of the tensor-core passes (csrc/host_digits.cpp) on the CPU: the blocks, decoded from their 64-byte swizzled
rows, give the half-size matrices back: FP64 as seven balanced base-256 digits on a common exponent per row, with every
column in the same binade, FP32 as two FP16 parts; what lies beyond the matrix is zero."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
DP = np.ctypeslib.ndpointer(dtype=np.float64, flags="C_CONTIGUOUS")
IP = np.ctypeslib.ndpointer(dtype=np.int32, flags="C_CONTIGUOUS")
BP = np.ctypeslib.ndpointer(dtype=np.uint8, flags="C_CONTIGUOUS")
D, NC, NC32 = 7, 32, 64
SIZES = [1, 2, 16, 31, 32, 33, 50, 64, 65, 127, 128]

WRAP = r"""
#include <cstring>
#include "fv_internal.h"
namespace fv { void set_error(const std::string&) {} }
static_assert(fv::kDigits64 == 7 && fv::kDigitCols64 == 32 && fv::kDigitCols32 == 64 && fv::kDigitMaxColumn == 48, "");
static long long give(const std::vector<unsigned char>& b, const std::vector<int>& e, unsigned char* blocks, int* exps) {
  std::memcpy(blocks, b.data(), b.size());
  std::memcpy(exps, e.data(), 4 * e.size());
  return (long long)b.size();
}
extern "C" long long digits(int h, int shared, const double* M0, const double* M1, unsigned char* blocks, int* exps,
                            unsigned char* cexps) {
  const std::vector<double> M[2] = {std::vector<double>(M0, M0 + h * h), std::vector<double>(M1, M1 + h * h)};
  std::vector<unsigned char> b, c;
  std::vector<int> e;
  fv::build_digits(M, h, fv::kDigits64, fv::kDigitCols64, shared != 0, b, e, c);
  std::memcpy(cexps, c.data(), c.size());
  return give(b, e, blocks, exps);
}
extern "C" int reached(int nx, int ny, int nz, int prec) {
  const int n[3] = {nx, ny, nz};
  return fv::digits_reached(n, prec);
}
extern "C" long long halves(int h, const double* M0, const double* M1, unsigned char* blocks, int* exps) {
  const std::vector<double> M[2] = {std::vector<double>(M0, M0 + h * h), std::vector<double>(M1, M1 + h * h)};
  std::vector<unsigned char> b;
  std::vector<int> e;
  fv::build_halves(M, h, fv::kDigitCols32, b, e);
  return give(b, e, blocks, exps);
}
"""


@pytest.fixture(scope="module")
def L(tmp_path_factory):
    d = tmp_path_factory.mktemp("digits")
    src, out = d / "wrap.cpp", d / "libdigits.so"
    src.write_text(WRAP)
    csrc = os.path.join(ROOT, "paper_2210_08816_gb300", "csrc")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f"-I{cuda}/include", f"-I{csrc}", str(src),
                        os.path.join(csrc, "host_digits.cpp"), "-o", str(out)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = C.CDLL(str(out))
    lib.digits.restype = lib.halves.restype = C.c_longlong
    lib.digits.argtypes = [C.c_int, C.c_int, DP, DP, BP, IP, BP]
    lib.halves.argtypes = [C.c_int, DP, DP, BP, IP]
    return lib


def _matrices(h, span):
    """Two matrices whose rows and columns span 2^span, with zeros, a zero column and exact powers of two."""
    rng = np.random.default_rng(100 * h + span)
    r, c = np.exp2(rng.integers(-span, span + 1, h)), np.exp2(rng.integers(-span, span + 1, h))
    M = [rng.standard_normal((h, h)) * r[:, None] * c[None, :] for _ in range(2)]
    M[0][rng.random((h, h)) < 0.1] = 0.0
    M[1][0, 0] = -np.exp2(float(span))
    if h > 2:
        M[1][:, h - 1] = 0.0  # the slot a shorter part leaves over
        M[1][h - 1] = 0.0
    return [np.ascontiguousarray(m) for m in M]


def _decode(blocks, h, parts, cols):
    """[matrix][part of the value][output][input], padded to whole groups and slabs."""
    groups, nslab = -(-h // cols), -(-h // 32)
    x = blocks.view(np.float16).astype(np.float64).reshape(2, groups, nslab, parts * cols, 4, 8)
    r = np.arange(parts * cols)
    out = np.empty_like(x)
    for c in range(4):
        out[:, :, :, r, c] = x[:, :, :, r, c ^ ((r >> 1) & 3)]
    out = out.reshape(2, groups, nslab, parts, cols, 32).transpose(0, 3, 1, 4, 2, 5)
    return out.reshape(2, parts, groups * cols, nslab * 32)


def _size(h, parts, cols):
    return 2 * (-(-h // cols)) * (-(-h // 32)) * parts * cols * 64


@pytest.mark.parametrize("h", SIZES)
@pytest.mark.parametrize("span", [0, 12])
@pytest.mark.parametrize("shared", [0, 1])
def test_digits_give_the_matrices_back(L, h, span, shared):
    M = _matrices(h, span)
    blocks, exps, cexps = np.zeros(_size(h, D, NC), np.uint8), np.zeros(h, np.int32), np.zeros(2 * h, np.uint8)
    assert L.digits(h, shared, M[0], M[1], blocks, exps, cexps) == blocks.size
    dig = _decode(blocks, h, D, NC)
    assert np.array_equal(dig, np.rint(dig)) and np.max(np.abs(dig)) <= 128
    assert not dig[:, :, h:].any() and not dig[:, :, :, h:].any()
    c = cexps.reshape(2, h).astype(int)
    top = 0
    for part in range(2):
        J = np.zeros((h, h), dtype=object)
        for i in range(D):
            J = J * 256 + np.vectorize(int, otypes=[object])(dig[part, i, :h, :h])
        scaled = np.ldexp(M[part], c[part][None, :])
        for j in range(h):  # rounded to the nearest unit 2^exps
            want = [int(np.rint(np.ldexp(v, -int(exps[j])))) for v in scaled[j]]
            assert list(J[j]) == want
        top = np.maximum(top, np.array([max(abs(int(v)) for v in row) for row in J], dtype=object))
    for j in range(h):  # every row with an entry fills its 55 bits
        assert top[j] == 0 or 2 ** 54 <= top[j] <= 2 ** 55
    # every column's largest entry lies in the same binade
    most = np.stack([np.abs(np.ldexp(M[p], c[p][None, :])).max(0) for p in range(2)])
    if shared:
        assert np.array_equal(c[0], c[1])
        most = most.max(0, keepdims=True)
    e = np.frexp(most[most > 0])[1]
    assert np.all(e == e.max())


def test_column_exponents_are_bounded(L):
    M = [np.ascontiguousarray(np.diag(np.exp2([0.0, -30.0, -60.0, -300.0]))) for _ in range(2)]
    blocks, exps, cexps = np.zeros(_size(4, D, NC), np.uint8), np.zeros(4, np.int32), np.zeros(8, np.uint8)
    L.digits(4, 1, M[0], M[1], blocks, exps, cexps)
    assert list(cexps) == [0, 30, 48, 48] * 2


@pytest.mark.parametrize("h", SIZES)
@pytest.mark.parametrize("span", [0, 12])
def test_halves_give_the_matrices_back(L, h, span):
    M = _matrices(h, span)
    blocks, exps = np.zeros(_size(h, 2, NC32), np.uint8), np.zeros(h, np.int32)
    assert L.halves(h, M[0], M[1], blocks, exps) == blocks.size
    v = _decode(blocks, h, 2, NC32)
    assert not v[:, :, h:].any() and not v[:, :, :, h:].any()
    for part in range(2):
        x = np.ldexp(M[part], -exps[:, None])
        assert np.max(np.abs(x)) < 2.0 ** 14
        hi = x.astype(np.float16).astype(np.float64)
        assert np.array_equal(v[part, 0, :h, :h], hi)
        assert np.array_equal(v[part, 1, :h, :h], (x - hi).astype(np.float16).astype(np.float64))
        err = np.abs(v[part].sum(0)[:h, :h] - x)
        assert np.all(err <= np.maximum(2.0 ** -22 * np.abs(x), 2.0 ** -25))


@pytest.mark.parametrize("n,want64,want32", [
    ((2, 2, 2), 0, 0), ((8, 8, 8), 0, 0), ((16, 16, 16), 0, 0), ((31, 31, 31), 0, 0), ((32, 32, 32), 0, 1), ((35, 35, 35), 0, 0),
    ((36, 36, 36), 1, 0), ((40, 41, 42), 1, 0), ((17, 33, 65), 1, 0), ((16, 16, 256), 1, 1), ((12, 12, 255), 1, 0),
    ((4, 4, 255), 0, 0), ((55, 55, 55), 1, 0), ((57, 57, 57), 1, 1), ((64, 64, 64), 1, 1)])
def test_operands_are_made_where_a_pass_takes_them(L, n, want64, want32):
    """A pass of four fields along the longest axis makes 4 N ceil(n / 2) multiplications and takes the digits from 3.2e6 on,
    the FP32 parts from 2e7; axes of a multiple of 32 cells, 32 to 256, take the FP32 pressure passes."""
    work = 4.0 * n[0] * n[1] * n[2] * ((max(n) + 1) // 2)
    tc = all(32 <= k <= 256 and k % 32 == 0 for k in n)
    assert L.reached(*n, 0) == int(work >= 3.2e6)
    assert L.reached(*n, 1) == int(work >= 2.0e7 or tc)
    assert (L.reached(*n, 0), L.reached(*n, 1)) == (want64, want32)
