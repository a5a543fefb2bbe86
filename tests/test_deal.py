"""The batched product's deal of units to blocks, checked on the host for every
layout shape (tests/c/deal_check.cpp against csrc/vbq_deal.h): above all, no
block waits for the zeroed rows of a block after it, so a launch that shares
the GPU with another stream's kernels never waits on a block that may have no
room to start. CPU only."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_deal_of_units(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "deal_check")
    cmd = [cxx, "-std=c++17", "-O2", "-Wall", "-Wextra", "-Werror", "-I", os.path.join(ROOT, "paper_2607_02893_gb300", "csrc"),
           os.path.join(ROOT, "tests", "c", "deal_check.cpp"), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, f"compile failed:\n{r.stdout}\n{r.stderr}"
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "ALL OK" in r.stdout, r.stdout + r.stderr
