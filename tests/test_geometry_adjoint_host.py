"""Host memory of the reverse-mode geometry (CPU): what a shape gradient allocates does not grow with
the cores that work on it, and neither does its result change."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_1812_00394_gb300", "csrc")


def test_geometry_adjoint_memory_does_not_depend_on_the_threads(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "geometry_adjoint_memory")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-fopenmp", "-I", os.path.join(ROOT, "include"),
                           "-I", CSRC, os.path.join(HERE, "native", "geometry_adjoint_memory.cpp"),
                           os.path.join(CSRC, "fvlbm_host.cpp"), "-o", exe])

    def run(threads):
        env = dict(os.environ, OMP_NUM_THREADS=str(threads), OMP_DYNAMIC="false")
        return subprocess.run([exe, "40"], capture_output=True, text=True, check=True, env=env).stdout

    assert run(1) == run(8)
