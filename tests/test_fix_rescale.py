"""CPU check of the exponents of lines in fixed point (csrc/fix_fft.h), compiled
with g++: bounds of a line brought to one unit."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_rescaled_lines(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    exe = tmp_path / "fix_rescale_check"
    subprocess.run([gxx, "-O2", "-std=c++17", "-Wall", "-I",
                    os.path.join(ROOT, "paper_2102_01031_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "fix_rescale_check.cpp"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.startswith("OK"), r.stdout
