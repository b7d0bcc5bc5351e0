"""Build the CUDA library libcubefv.so in-tree for sm_103a (GB300).

Each translation unit is compiled by nvcc in parallel (one -gencode, -O3, -lineinfo) into
_build/, then linked into _lib/libcubefv.so.  Objects newer than their sources and headers are
reused.  No cmake, no torch headers: the library is plain CUDA C++ behind a C ABI.
"""
from __future__ import annotations

import os
import shutil
import subprocess
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "_build")
LIBDIR = os.path.join(HERE, "_lib")
LIB = os.path.join(LIBDIR, "libcubefv.so")
SOURCES = ["kernels_stencil.cu", "kernels_stencil2.cu", "kernels_flux.cu", "kernels_fdm.cu", "kernels_tc.cu", "kernels_plane.cu", "kernels_digit.cu", "kernels_blas.cu", "host_linalg.cpp",
           "host_cheb.cpp", "host_grid.cpp", "host_digits.cpp", "fv_api.cpp", "noalloc.cu", "kernels_prolong.cu", "kernels_diag.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def _nvcc() -> str:
    for c in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", shutil.which("nvcc")):
        if c and os.path.exists(c):
            return c
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libcubefv.so")


def _headers():
    return [os.path.join(CSRC, "fv_internal.h"), os.path.join(CSRC, "tcgen05.cuh"), os.path.join(CSRC, "launch.cuh"), os.path.join(ROOT, "include", "cube_fv.h")]


def _stale(obj: str, deps) -> bool:
    if not os.path.exists(obj):
        return True
    t = os.path.getmtime(obj)
    return any(os.path.getmtime(d) > t for d in deps)


def build(verbose: bool = False, force: bool = False, extra_flags=()) -> str:
    nvcc = _nvcc()
    os.makedirs(OBJ, exist_ok=True)
    os.makedirs(LIBDIR, exist_ok=True)
    common = [*ARCH, "-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC,-O2", "--expt-relaxed-constexpr",
              "-I", os.path.join(ROOT, "include"), *extra_flags]
    jobs = []
    for src in SOURCES:
        s = os.path.join(CSRC, src)
        o = os.path.join(OBJ, os.path.splitext(src)[0] + ".o")
        if force or _stale(o, [s, *_headers()]):
            jobs.append([nvcc, *common, "-c", s, "-o", o])

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed:\n" + " ".join(cmd) + "\n" + r.stdout + r.stderr)
        if verbose and (r.stdout or r.stderr):
            print(r.stdout + r.stderr)

    with ThreadPoolExecutor(max_workers=max(1, min(len(SOURCES), os.cpu_count() or 1))) as ex:
        list(ex.map(run, jobs))
    objs = [os.path.join(OBJ, os.path.splitext(s)[0] + ".o") for s in SOURCES]
    if force or jobs or not os.path.exists(LIB):
        tmp = LIB + ".tmp"
        run([nvcc, *ARCH, "-shared", "-o", tmp, *objs])
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    import sys
    print(build(verbose=True, force="--force" in sys.argv))
