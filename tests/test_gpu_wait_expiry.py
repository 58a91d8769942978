"""Waits of the tensor-core GEMMs (jamp_gemm.cu, colour_gemm.cu) that run out: a
launch whose waits expire, at once or somewhere on the way, ends by itself with
its status word set and leaves the context usable
(tests/native/wait_expiry.cu).  One column block with derived columns, one
without, and two blocks; two CTAs per SM and one in the colour sum."""
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
    procs = ["21,21,21,21,21,21", "2,-2,21,21,21,21", "2,2,2,2,21,21,21"]
    r = subprocess.run([exe] + procs, capture_output=True, text=True, timeout=240)
    assert r.returncode == 0, r.stdout + r.stderr
    rows = [line.split() for line in r.stdout.splitlines()[1:]]
    assert [row[0] for row in rows] == procs
    for name, amplitudes, total in rows:
        assert int(amplitudes) >= 1 and int(total) >= 1, name
