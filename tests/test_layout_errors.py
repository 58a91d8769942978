"""Layouts refuse a process with their own error type (tests/native/layout_errors_check.cpp);
any other exception of a layout is an error of the handle, not a silent fallback."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_0909_5257_gb300", "csrc")


def test_refused_layouts_raise_their_own_error(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "layout_errors_check")
    subprocess.run([cxx, "-O1", "-std=c++17", "-fopenmp", "-I", CSRC, "-o", exe,
                    os.path.join(HERE, "native", "layout_errors_check.cpp")] +
                   [os.path.join(CSRC, f) for f in ("phased.cpp", "ordered.cpp", "colour_base.cpp", "generator.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
