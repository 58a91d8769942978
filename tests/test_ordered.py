"""Host check of the ordered recursion (csrc/ordered.cpp, ordered_eval.cuh):
|M|^2 equals the sum over every Feynman diagram and helicity combination of
the per-lane program on phase-space points (tests/native/ordered_check.cpp)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_0909_5257_gb300", "csrc")


def test_ordered_recursion_gives_the_diagram_sum(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "ordered_check")
    subprocess.run([cxx, "-O1", "-std=c++17", "-fopenmp", "-I", CSRC, "-o", exe,
                    os.path.join(HERE, "native", "ordered_check.cpp")] +
                   [os.path.join(CSRC, f) for f in ("ordered.cpp", "colour_base.cpp", "generator.cpp")], check=True)
    procs = ["21,21,21,21", "21,21,21,21,21", "21,21,21,21,21,21", "21,21,21,21,21,21,21",
             "2,-2,21,21", "2,-2,21,21,21", "2,-2,21,21,21,21", "2,-2,21,21,21,21,21",
             "2,2,2,2", "2,2,2,2,21", "2,2,2,2,21,21", "2,2,2,2,21,21,21",
             # crossings and other flavours
             "2,1,2,1,21", "2,1,2,1,21,21,21", "2,-2,2,-2,21", "2,21,2,21", "21,2,2,21", "2,21,2,21,21", "2,21,2,21,21,21,21",
             "2,-2,1,-1,21", "2,-2,1,-1,21,21", "-1,-1,-1,-1,21", "21,-2,-2,21,21"]
    r = subprocess.run([exe] + procs, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    rows = [line.split() for line in r.stdout.splitlines()]
    assert [row[0] for row in rows] == procs
    for name, worst, area, amplitudes in rows:
        # sums of up to 1e4 products of rounded FP64 numbers
        assert float(worst) < 1e-13, name
