"""The profiler constants of bench.py are valid for the sources they were taken on: the hash
that guards each changes with every header that its kernel includes, directly or through another,
and with the header that splits its work."""
import os
import shutil

import pytest

import bench

CSRC = os.path.join(bench.ROOT, "paper_2102_01031_gb300", "csrc")
COMMON = ["common.cuh", "fix_fft.h", "friedmann.h", "tail.cuh", "worklist.h"]


@pytest.mark.parametrize("hash_of,names", [
    ("kernel_source_hash", COMMON + ["pass_scalar.cu", "ring.cuh", "fix_lap.h"]),
    ("u1_source_hash", COMMON + ["pass_u1.cu", "ring.cuh", "kd_drift.cuh", "trig2.cuh"]),
    ("su2_source_hash", COMMON + ["pass_su2_kd.cu", "su2_kick.cuh", "su2_common.cuh", "su2_work.h", "kd_drift.cuh",
                                  "trig2.cuh"]),
])
def test_source_hash_covers_every_header(hash_of, names, tmp_path, monkeypatch):
    copy = tmp_path / "paper_2102_01031_gb300" / "csrc"
    shutil.copytree(CSRC, copy)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    f = getattr(bench, hash_of)
    seen = {f()}
    for name in names:
        with open(copy / name, "a") as h:
            h.write("\n// changed\n")
        assert f() not in seen, name
        seen.add(f())
    with open(copy / "probe.cu", "a") as h:  # a file that the pass has nothing to do with
        h.write("\n// changed\n")
    assert f() in seen
