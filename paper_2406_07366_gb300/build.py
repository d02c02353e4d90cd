"""Build the CUDA library ``libbsewald.so`` in-tree with nvcc for sm_103a.

Each translation unit is compiled in parallel into ``_build/`` and linked
with cuFFT into ``paper_2406_07366_gb300/lib/libbsewald.so``.  Nothing is
installed into site-packages.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(ROOT, "_build")
LIBDIR = os.path.join(PKG, "lib")
LIB = os.path.join(LIBDIR, "libbsewald.so")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
SOURCES = ["bs_api.cu", "k_geometry.cu", "k_sort.cu", "k_short.cu", "k_long.cu", "k_fft.cu", "k_static_short.cu", "k_rk4.cu",
           "k_peak.cu"]
# sources compiled again with macros: the transform kernels, an object per precision for the single
# contexts and one for the batches
VARIANTS = [("k_fft.cu", "k_fft_f64.o", ["-DBSW_FFT_DOUBLE"]), ("k_fft.cu", "k_fft_b.o", ["-DBSW_FFT_BATCH"]),
            ("k_fft.cu", "k_fft_f64_b.o", ["-DBSW_FFT_DOUBLE", "-DBSW_FFT_BATCH"])]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _cuda_lib_dir(nvcc: str) -> str:
    root = os.path.dirname(os.path.dirname(os.path.realpath(nvcc)))
    for sub in ("lib64", "lib", "targets/sbsa-linux/lib", "targets/x86_64-linux/lib"):
        d = os.path.join(root, sub)
        if os.path.exists(os.path.join(d, "libcufft.so")):
            return d
    return os.path.join(root, "lib64")


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build_library(verbose: bool = False, extra_flags=None, force: bool = False) -> str:
    """Compile every .cu file for sm_103a and link libbsewald.so; return its path."""
    nvcc = _nvcc()
    os.makedirs(BUILD, exist_ok=True)
    os.makedirs(LIBDIR, exist_ok=True)
    headers = [os.path.join(CSRC, "bs_internal.cuh"), os.path.join(INCLUDE, "bsewald.h")]
    flags = ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC,
                    "--expt-relaxed-constexpr"] + list(extra_flags or [])
    objs, jobs = [], []
    units = [(src, src.replace(".cu", ".o"), []) for src in SOURCES] + VARIANTS
    for src, obj, extra in sorted(units, key=lambda u: u[0] != "k_fft.cu"):  # the longest first
        s = os.path.join(CSRC, src)
        o = os.path.join(BUILD, obj)
        objs.append(o)
        if force or _stale(o, [s] + headers):
            jobs.append([nvcc, "-c", s, "-o", o] + flags + extra)

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed:\n" + " ".join(cmd) + "\n" + r.stdout + r.stderr)
        if verbose and (r.stdout or r.stderr):
            sys.stderr.write(r.stdout + r.stderr)

    if jobs:
        with cf.ThreadPoolExecutor(max_workers=min(len(jobs), os.cpu_count() or 4)) as ex:
            list(ex.map(run, jobs))
    if force or jobs or _stale(LIB, objs):
        libdir = _cuda_lib_dir(nvcc)
        tmp = LIB + f".tmp{os.getpid()}"
        run([nvcc] + ARCH + ["-shared", "-o", tmp] + objs +
            ["-L", libdir, "-lcufft", "-lcudart", "-Xlinker", "-rpath," + libdir])
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build_library(verbose="-v" in sys.argv, force="-f" in sys.argv))
