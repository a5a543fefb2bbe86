"""The error words of the validating calls, checked on the host against a fake
CUDA runtime (tests/c/error_words_check.cpp): several devices, one of them
reset, many threads, more live calls than the page has lines. CPU only."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def cuda_include():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    return os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")


def test_error_words(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    if not os.path.exists(os.path.join(cuda_include(), "cuda_runtime_api.h")):
        pytest.skip("no CUDA headers")
    exe = str(tmp_path / "error_words_check")
    cmd = [cxx, "-std=c++17", "-O1", "-Wall", "-Wextra", "-Werror", "-pthread", "-isystem", cuda_include(),
           "-I", os.path.join(ROOT, "paper_2607_02893_gb300", "csrc"),
           os.path.join(ROOT, "tests", "c", "error_words_check.cpp"), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, f"compile failed:\n{r.stdout}\n{r.stderr}"
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "ALL OK" in r.stdout, r.stdout + r.stderr
