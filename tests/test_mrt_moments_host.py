"""The fixed-point moments of the MRT collision on the host: no arithmetic that the language leaves
undefined for any population (densities of 32 to 38 pass the test of each population), exact
moments for the nodes it takes, and no other node taken."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_fixed_point_moments(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "mrt_host_check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-fsanitize=undefined", "-fno-sanitize-recover=all",
                    "-o", exe, os.path.join(ROOT, "tests", "mrt_host_check.cpp")], check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr
    got = {k: int(v) for k, v in (line.split() for line in r.stdout.splitlines())}
    assert got["taken"] > 50000 and got["wide"] > 50000
    assert got["wrong_choice"] == 0 and got["wrong_moment"] == 0
