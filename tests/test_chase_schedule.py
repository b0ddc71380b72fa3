"""The chase's schedule, walked on the host (tests/c/chase_walk.cpp): no
rotation record names a row or column outside the matrix, whatever values the
band holds.  The applies index their slabs with these records."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_records_stay_inside_the_matrix(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = tmp_path / "chase_walk"
    cmd = [gxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-I",
           os.path.join(ROOT, "paper_2509_02840_gb300", "csrc"), os.path.join(ROOT, "tests", "c", "chase_walk.cpp"),
           "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
