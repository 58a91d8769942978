"""The server ranks and cuts requests by an estimated cost per event: for the five-jet
processes, mixed and FP64, it follows the measured device times within a factor of 2
(tests/native/request_cost_check.cpp)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_estimated_costs_follow_the_measured_times(tmp_path):
    from paper_0909_5257_gb300 import build
    if shutil.which("g++") is None:
        pytest.skip("no host C++ compiler")
    lib = build.build()
    cuda = os.path.dirname(os.path.dirname(build.nvcc()))
    exe = str(tmp_path / "request_cost_check")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", build.CSRC, "-I", os.path.join(cuda, "include"), "-o", exe,
                    os.path.join(HERE, "native", "request_cost_check.cpp"), lib, "-Wl,-rpath=" + os.path.dirname(lib)], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
