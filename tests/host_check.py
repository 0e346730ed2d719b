"""Compiles a small C++ program against the library's host headers and runs it (no GPU, no CUDA library)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def run_host_program(source: str, folder) -> str:
    """Standard output of the program; the test fails if it does not compile or exits with an error."""
    cxx, nvcc = shutil.which("g++"), shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if cxx is None or not os.path.exists(os.path.join(include, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src, exe = os.path.join(folder, "check.cpp"), os.path.join(folder, "check")
    with open(src, "w") as f:
        f.write(source)
    r = subprocess.run([cxx, "-O2", "-std=c++17", "-pthread", "-I", include, "-I", os.path.join(ROOT, "include"),
                        "-I", os.path.join(ROOT, "paper_2010_14058_gb300", "csrc"), src, "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout
