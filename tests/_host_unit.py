"""Host parts of the library compiled by themselves: a small C++ program that includes them, with CUDA runtime functions
of its own in place of the runtime library (no GPU)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1611_04214_gb300", "csrc")


def run_host_unit(tmp_path, program: str, sources=()) -> str:
    """Compile `program` (and the named files of csrc) with g++ and return what it prints."""
    cxx = shutil.which("g++")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if cxx is None or not os.path.exists(os.path.join(include, "cuda_runtime_api.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    src = tmp_path / "unit.cpp"
    src.write_text(program)
    exe = str(tmp_path / "unit")
    cmd = [cxx, "-std=c++17", "-O1", "-I", CSRC, "-I", include, str(src), *[os.path.join(CSRC, s) for s in sources], "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-4000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)
    return r.stdout
