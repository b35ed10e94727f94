"""CPU check of the work split of partly filled tiles (csrc/worklist.h), compiled
with g++: every plane once, over sizes, tile heights and CTA counts."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_partly_filled_tiles(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    exe = tmp_path / "partial_tiles_check"
    subprocess.run([gxx, "-O2", "-std=c++17", "-Wall", "-I",
                    os.path.join(ROOT, "paper_2102_01031_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "partial_tiles_check.cpp"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.startswith("OK"), r.stdout
