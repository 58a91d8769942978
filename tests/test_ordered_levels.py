"""Host check of the ordered recursion's levels (tests/native/ordered_levels_check.cpp),
up to the largest processes: nothing that a level writes is read in it, so the CTA's
barriers stand where they are needed."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_0909_5257_gb300", "csrc")


def test_items_of_a_level_run_in_any_order(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "ordered_levels_check")
    subprocess.run([cxx, "-O1", "-std=c++17", "-fopenmp", "-I", CSRC, "-o", exe,
                    os.path.join(HERE, "native", "ordered_levels_check.cpp")] +
                   [os.path.join(CSRC, f) for f in ("ordered.cpp", "colour_base.cpp", "generator.cpp")], check=True)
    procs = ["21,21,21,21,21", "21,21,21,21,21,21", "21,21,21,21,21,21,21", "2,-2,21,21", "2,-2,21,21,21,21", "2,-2,21,21,21,21,21",
             "2,2,2,2", "2,2,2,2,21,21", "2,2,2,2,21,21,21", "2,1,2,1,21,21,21", "2,-2,2,-2,21,21,21", "2,21,2,21,21,21,21",
             "21,2,2,21,21,21", "2,-2,1,-1,21,21,21", "21,-2,-2,21,21"]
    r = subprocess.run([exe] + procs, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    assert [line.split()[0] for line in r.stdout.splitlines()] == procs
