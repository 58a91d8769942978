"""Host check of the phased layout (csrc/phased.cpp): its units, run phase by
phase in FP64, give every diagram amplitude of every summed helicity
combination exactly once and bit for bit as the per-lane program, inside the
area, reading nothing the same phase writes (tests/native/phased_check.cpp)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_0909_5257_gb300", "csrc")


def test_phased_layout_gives_the_per_lane_amplitudes(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "phased_check")
    subprocess.run([cxx, "-O1", "-std=c++17", "-fopenmp", "-ffp-contract=off", "-I", CSRC, "-o", exe,
                    os.path.join(HERE, "native", "phased_check.cpp"), os.path.join(CSRC, "phased.cpp"),
                    os.path.join(CSRC, "generator.cpp")], check=True)
    procs = ["21,21,21,21,21,21,21", "2,-2,21,21,21,21,21", "2,2,2,2,21,21,21", "21,21,21,21,21,21", "2,-2,21,21,21,21",
             "2,2,2,2,21,21",
             # crossings and other flavours
             "2,21,2,21,21,21,21", "2,-2,2,-2,21,21,21", "2,1,2,1,21,21,21", "21,2,2,21,21,21", "2,-2,1,-1,21,21"]
    r = subprocess.run([exe] + procs, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    rows = [line.split() for line in r.stdout.splitlines()]
    assert [row[0] for row in rows] == procs
    for name, compared, mismatched, area in rows:
        assert int(compared) > 0 and int(mismatched) == 0, name
        assert 32 * int(area) < 200 * 1024, name  # fits a CTA's shared memory
    # half of the 112 combinations of g g -> 5g: the flipped ones are conjugate
    assert int(rows[0][1]) == 56 * 7245
