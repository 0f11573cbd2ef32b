"""Build the in-tree shared library ``libmolt.so`` for sm_103a with nvcc.

The translation units are compiled in parallel and linked with the static CUDA runtime, so the
library needs only the NVIDIA driver at run time.  Usage: ``python -m paper_1611_04214_gb300.build``.
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG, "csrc")
ROOT = os.path.dirname(PKG)
LIB = os.path.join(PKG, "libmolt.so")
BUILD_DIR = os.path.join(ROOT, "_build")
SOURCES = ["kernels_f32.cu", "kernels_f64.cu", "kernels_p1.cu", "kernels_p2.cu", "kernels_p3.cu", "kernels_p4.cu",
           "kernels_v1.cu", "kernels_v2.cu", "kernels_c3.cu", "kernels_vch_f32.cu", "kernels_vch_f64.cu", "line_params.cpp", "solver.cpp",
           "noalloc.cu", "batch.cu", "selftest.cu", "probe.cu", "rows_tc.cu", "solver3d.cpp",
           "nest.cpp", "nest_f32_m2.cu", "nest_f32_m4.cu", "nest_f32_m6.cu", "nest_f64_m2.cu", "nest_f64_m4.cu",
           "nest_f64_m6.cu", "nest_line.cu", "fch1d.cpp", "fch2d.cpp"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-std=c++17", "-O3", "-lineinfo", "-Xcompiler", "-fPIC,-O2", "-I", os.path.join(ROOT, "include")]


def _nvcc() -> str:
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found: the CUDA 13 toolkit is required to build libmolt.so")
    return exe


def _stale(objs) -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(ROOT, "include", "molt.h")]
    return any(os.path.getmtime(p) > t for p in deps)


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compile and link ``libmolt.so`` (skipped when it is newer than every source)."""
    os.makedirs(BUILD_DIR, exist_ok=True)
    objs = [os.path.join(BUILD_DIR, os.path.splitext(s)[0] + ".o") for s in SOURCES]
    if not force and not _stale(objs):
        return LIB
    nvcc = _nvcc()

    def compile_one(src_obj):
        src, obj = src_obj
        cmd = [nvcc, *ARCH, *FLAGS, "-c", os.path.join(CSRC, src), "-o", obj]
        if src.endswith(".cpp"):
            cmd = [nvcc, *FLAGS, "-x", "c++", "-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
        if verbose:
            sys.stdout.write(r.stdout + r.stderr)
        return obj

    with ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        list(ex.map(compile_one, zip(SOURCES, objs)))
    tmp = LIB + ".tmp"
    cmd = [nvcc, *ARCH, "-shared", "-cudart", "static", "-o", tmp, *objs]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose="-v" in sys.argv))
