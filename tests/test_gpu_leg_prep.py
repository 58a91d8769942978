"""FP64 gluon polarisation bases are correctly rounded roots and quotients
(tests/native/leg_prep.cu): the FP64 path's accuracy starts there."""
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_fp64_polarisation_bases_are_correctly_rounded(tmp_path):
    from paper_0909_5257_gb300 import build
    exe = str(tmp_path / "leg_prep")
    subprocess.run([build.nvcc()] + build.ARCH + ["-O3", "-std=c++17", "-I", build.CSRC, "-o", exe,
                    os.path.join(HERE, "native", "leg_prep.cu")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
