"""Small straight-line calls spread over the SMs of the handle's own device
(tests/native/spread_check.cpp), whichever device was asked about first."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_tiles_follow_the_handles_device(tmp_path):
    from paper_0909_5257_gb300 import build
    if shutil.which("g++") is None:
        pytest.skip("no host C++ compiler")
    lib = build.build()
    cuda = os.path.dirname(os.path.dirname(build.nvcc()))
    exe = str(tmp_path / "spread_check")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", build.CSRC, "-I", os.path.join(cuda, "include"), "-o", exe,
                    os.path.join(HERE, "native", "spread_check.cpp"), lib, "-Wl,-rpath=" + os.path.dirname(lib)], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
