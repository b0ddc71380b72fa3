"""The chase's schedule and watchdog on the host.  tests/c/chase_walk.cpp walks
the schedule: no rotation record names a row or column outside the matrix,
whatever values the band holds (the applies index their slabs with these
records).  tests/c/chase_waits.cpp holds the poll limits against what a wait
may last."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("name", ["chase_walk", "chase_waits"])
def test_on_the_host(tmp_path, name):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = tmp_path / name
    cmd = [gxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-I",
           os.path.join(ROOT, "paper_2509_02840_gb300", "csrc"), os.path.join(ROOT, "tests", "c", name + ".cpp"),
           "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
