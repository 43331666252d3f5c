"""Blocks dealt to the kinds of a batch's members (host logic, no GPU).  The check
is a small C++ program linked against the built library."""
import os
import shutil
import subprocess

import pytest

from paper_1603_09255_gb300 import build as pkg_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_blocks_are_dealt_by_work(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no host C++ compiler")
    pkg_build.build()
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    exe = str(tmp_path / "deal_check")
    cmd = ["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-I", pkg_build.CSRC, "-I", cuda,
           os.path.join(ROOT, "tests", "deal_check.cpp"), "-L", pkg_build.OUT_DIR, "-lspegg_gb300",
           "-Wl,-rpath," + pkg_build.OUT_DIR, "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.rstrip().endswith("ok"), r.stdout[-2000:]
