"""Planned residency of the straight-line kernels is the runtime's for kernels that
were never launched (tests/native/resident_check.cu), so a plan does not depend on
what an earlier handle launched."""
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_residency_is_the_runtimes(tmp_path):
    from paper_0909_5257_gb300 import build
    lib = build.build()
    exe = str(tmp_path / "resident_check")
    subprocess.run([build.nvcc()] + build.ARCH + ["-cudart", "shared", "-O1", "-std=c++17", "-I", build.CSRC, "-o", exe,
                    os.path.join(HERE, "native", "resident_check.cu"), lib, "-Xlinker", "-rpath=" + os.path.dirname(lib)], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
