"""The rules that cut a grid's planes into chunks (each_chunk, stencil_chunk) on the CPU: the same choice as by trying every
number of chunks, in a time that does not go by the number of planes (they run on every launch of a stencil)."""
import ctypes as C
import os
import subprocess
import time

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

WRAP = r"""
#include "fv_internal.h"
namespace fv { void set_error(const std::string&) {} }
static const fv::PlaneTimes kTimes[2] = {{2, {10, 17, 0}}, {3, {10, 16, 23}}};
extern "C" int chunk(int nz, int sms, int tiles, int nvec, int form) {
  return fv::stencil_chunk(nz, sms, tiles, nvec, kTimes[form]);
}
extern "C" int chunks(int nz, int* zc, int* n) {
  int k = 0;
  fv::each_chunk(nz, [&](int z, int c) { zc[k] = z; n[k++] = c; return true; });
  return k;
}
extern "C" long long many(int nz, int sms, int tiles, int nvec, int times) {
  long long s = 0;
  for (int i = 0; i < times; ++i) s += fv::stencil_chunk(nz, sms, tiles + (i & 1), nvec, kTimes[i & 1]);
  return s;
}
"""


@pytest.fixture(scope="module")
def L(tmp_path_factory):
    d = tmp_path_factory.mktemp("chunks")
    src, out = d / "wrap.cpp", d / "libchunks.so"
    src.write_text(WRAP)
    csrc = os.path.join(ROOT, "paper_2210_08816_gb300", "csrc")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f"-I{cuda}/include", f"-I{csrc}", str(src),
                        os.path.join(csrc, "host_grid.cpp"), os.path.join(csrc, "host_linalg.cpp"), "-o", str(out)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = C.CDLL(str(out))
    lib.many.restype = C.c_longlong
    return lib


def test_every_distinct_cut_once(L):
    zc, n = np.zeros(2048, np.int32), np.zeros(2048, np.int32)
    p = lambda a: a.ctypes.data_as(C.POINTER(C.c_int))  # noqa: E731
    for nz in [*range(1, 200), 255, 256, 257, 500, 811, 812]:
        k = L.chunks(nz, p(zc), p(n))
        want = [(-(-nz // c), c) for c in range(1, nz + 1) if -(-nz // -(-nz // c)) == c]
        assert list(zip(zc[:k].tolist(), n[:k].tolist())) == want
        assert k <= 2 * np.sqrt(nz) + 1


TIMES = [(10, 17), (10, 16, 23)]


def _tried(nz, sms, tiles, nvec, t):
    best, cost = nz, None
    for c in range(1, nz + 1):
        zc = -(-nz // c)
        n = -(-nz // zc)
        if tiles * n * nvec > 1 << 20 or n * nvec > 65535:
            break
        waves, rest = divmod(-(-(tiles * n * nvec) // sms), len(t))
        now = (waves * t[-1] + (t[rest - 1] if rest else 0)) * (zc + 1)
        if cost is None or now < cost:
            best, cost = zc, now
    return best


def test_the_choice_is_that_of_trying_all(L):
    rng = np.random.default_rng(1)
    cases = [(nz, t, v) for nz in (1, 2, 5, 16, 64, 100, 256, 812) for t in (1, 4, 16, 128, 700) for v in (1, 2, 16, 333)]
    cases += [tuple(int(x) for x in np.exp(rng.uniform(0, np.log([812, 2000, 70000])))) for _ in range(300)]
    for nz, tiles, nvec in cases:
        for form, t in enumerate(TIMES):
            assert L.chunk(nz, 152, tiles, nvec, form) == _tried(nz, 152, tiles, nvec, t), (nz, tiles, nvec)


# the fastest cuts as timed on 152 multiprocessors, and what was chosen when planes alone counted
@pytest.mark.parametrize("form,nz,tiles,nvec,good,bad", [
    (0, 192, 72, 1, (48, 24), 96), (0, 64, 8, 6, (11,), 22), (0, 32, 16, 8, (7, 16), 32),
    (1, 96, 36, 2, (16, 9, 8), 48), (1, 32, 4, 33, (16, 4), 32), (1, 256, 4, 3, (7, 11), 22)])
def test_large_grids_are_not_left_with_one_block_per_multiprocessor(L, form, nz, tiles, nvec, good, bad):
    zc = L.chunk(nz, 152, tiles, nvec, form)
    assert zc in good and zc != bad


def test_the_time_does_not_go_by_the_planes(L):
    def seconds(nz):
        best = 1e9
        for _ in range(5):
            t = time.perf_counter()
            L.many(nz, 152, 4, 2, 3000)
            best = min(best, time.perf_counter() - t)
        return best
    assert seconds(800) <= 30.0 * seconds(8)  # 57 cuts against 5; all of them would be 800 against 8
