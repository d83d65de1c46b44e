"""The library's critical t values over the whole range of alpha, on the host
(tests/tdist_range_check.cpp)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2408_07996_gb300", "csrc")


def test_critical_values_of_every_alpha_equal_bisection(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("g++ is missing")
    exe = str(tmp_path / "tdist_range_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, os.path.join(ROOT, "tests", "tdist_range_check.cpp"),
                    os.path.join(CSRC, "tdist.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    print(out.stdout.strip())
    assert out.returncode == 0 and out.stdout.startswith("OK"), out.stdout + out.stderr
