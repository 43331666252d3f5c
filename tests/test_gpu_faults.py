"""Waits and jobs that end with an error (see fault_check.cpp): a block of a team
that never arrives, or too late; a served job with an error status."""
import os
import shutil
import subprocess

import pytest

from paper_1603_09255_gb300 import build as pkg_build

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg_build.build()
    exe = str(tmp_path_factory.mktemp("fault") / "fault_check")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cmd = [nvcc, "-std=c++17", "-O1", "-cudart", "shared", "-I", os.path.join(ROOT, "include"), "-I", pkg_build.CSRC,
           os.path.join(ROOT, "tests", "fault_check.cpp"), "-L", pkg_build.OUT_DIR, "-lspegg_gb300",
           "-Xlinker", "-rpath," + pkg_build.OUT_DIR, "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    return exe


def run(program, what):
    r = subprocess.run([program, what], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.rstrip().endswith("ok"), r.stdout[-2000:] + r.stderr[-2000:]


def test_a_wait_that_runs_out_is_kept(program):
    """Nobody passes the barrier once a block has given up: the generation is
    not closed, the status stays, and a restored checkpoint starts afresh."""
    run(program, "barrier")


def test_a_failed_generation_leaves_no_locus_counts(program):
    """The counts of the restored run hold nothing of the generation that failed."""
    run(program, "counts")


def test_a_served_job_with_an_error_is_finished(program):
    """It gives back its memory, keeps its statistics and its status, and the
    other jobs run to their ends."""
    run(program, "served")


def test_a_read_without_host_memory(program):
    """No exception leaves the C ABI."""
    run(program, "memory")
