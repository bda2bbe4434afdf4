"""Host walk of the index map of the true-residual sweep (csrc/sweep.h, tests/sweep_map.cpp):
no lane loads outside the lattice, narrow tori included, and every vertex is owned once."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_load_of_the_sweep_is_inside_the_lattice(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no C++ compiler")
    from paper_1105_5256_gb300 import _build
    exe = str(tmp_path / "sweep_map")
    r = subprocess.run(["g++", "-std=c++17", "-O2", "-Wall", "-Werror", "-I", _build.CSRC, "-isystem",
                        os.path.join(_build._cuda_home(), "include"), os.path.join(ROOT, "tests", "sweep_map.cpp"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=30)
    assert r.returncode == 0, r.stdout
