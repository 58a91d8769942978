"""FP64 straight-line bodies (codegen.cpp) accumulate every colour amplitude from its
diagrams (tests/native/body_sums_check.cpp); sums of other colour amplitudes belong
to the compensated FP32 bodies."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_0909_5257_gb300", "csrc")


def test_fp64_bodies_sum_the_diagrams(tmp_path):
    from paper_0909_5257_gb300 import build
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    tool, gen = str(tmp_path / "codegen"), tmp_path / "generated"
    gen.mkdir()
    generator = str(tmp_path / "generator.o")
    subprocess.run([cxx, "-O1", "-std=c++17", "-fopenmp", "-c", "-o", generator, os.path.join(CSRC, "generator.cpp")], check=True)
    subprocess.run([cxx, "-O1", "-std=c++17", "-fopenmp", "-o", tool, generator] +
                   [os.path.join(CSRC, f) for f in ("codegen.cpp", "colour_base.cpp")], check=True)
    subprocess.run([tool, str(gen)] + build.GENERATED, check=True)
    for proc in build.GENERATED:
        name = "Body_p" + "".join("_m" + c[1:] if c[0] == "-" else "_" + c for c in proc.split(","))
        text = next(p for p in gen.iterdir() if p.name.endswith("_d_part_128.cu") and f"struct {name} " in p.read_text()).read_text()
        a = text.index("template <typename R>\nstruct")
        body = tmp_path / f"{name}.inc"
        body.write_text(text[a:text.index("\n};\n", a) + 4])
        exe = str(tmp_path / name)
        subprocess.run([cxx, "-O0", "-std=c++17", "-fopenmp", "-ffp-contract=off", "-I", CSRC, f'-DBODY_FILE="{body}"', f"-DBODY={name}",
                        "-o", exe, os.path.join(HERE, "native", "body_sums_check.cpp"), generator], check=True)
        r = subprocess.run([exe, proc], capture_output=True, text=True)
        assert r.returncode == 0, r.stdout + r.stderr
