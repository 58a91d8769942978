"""Registers of the straight-line u u~ -> g g body at the 128-register cap (compiled
here, ptxas' report): up to 96 keep 20 warps on an SM, 97 to 128 only 16, which
cost calls of 20000 events and more 12 to 33 %."""
import os
import re
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_0909_5257_gb300", "csrc")


def test_two_jet_quark_body_keeps_twenty_warps(tmp_path):
    from paper_0909_5257_gb300 import build
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    tool, gen = str(tmp_path / "codegen"), tmp_path / "generated"
    gen.mkdir()
    subprocess.run(["g++", "-O1", "-std=c++17", "-fopenmp", "-o", tool] +
                   [os.path.join(CSRC, f) for f in ("codegen.cpp", "colour_base.cpp", "generator.cpp")], check=True)
    subprocess.run([tool, str(gen), "2,-2,21,21"], check=True)
    for body in ("part", "diag"):
        src = gen / f"generated_p_2_m2_21_21_f_{body}_128.cu"
        r = subprocess.run([nvcc] + build.ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xptxas", "-v", "-I", CSRC, "-c", str(src),
                            "-o", str(tmp_path / "body.o")], check=True, capture_output=True, text=True)
        used = [int(x) for x in re.findall(r"Used (\d+) registers", r.stdout + r.stderr)]
        assert used and max(used) <= 96, used
        assert not re.search(r"[1-9]\d* bytes spill", r.stdout + r.stderr)
