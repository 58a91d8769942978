"""Waits of the tensor-core GEMMs that run out (tests/native/wait_expiry.cu): the
usual limit is a matter of seconds."""
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_expired_waits_end_the_launch(tmp_path):
    from paper_0909_5257_gb300 import build
    lib = build.build()
    exe = str(tmp_path / "wait_expiry")
    subprocess.run([build.nvcc()] + build.ARCH + ["-O1", "-std=c++17", "-I", build.CSRC, "-o", exe,
                    os.path.join(HERE, "native", "wait_expiry.cu"), lib,
                    "-Xlinker", "-rpath=" + os.path.dirname(lib)], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=240)
    assert r.returncode == 0, r.stdout + r.stderr
