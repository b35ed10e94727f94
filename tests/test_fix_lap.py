"""CPU check of the integer Laplacian sums of the FP64 passes (csrc/fix_lap.h), compiled
with g++: error against extended precision, the ends of the exponent range."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_integer_laplacian(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    exe = tmp_path / "fix_lap_check"
    subprocess.run([gxx, "-O2", "-std=c++17", "-Wall", "-I",
                    os.path.join(ROOT, "paper_2102_01031_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "fix_lap_check.cpp"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.startswith("OK"), r.stdout
