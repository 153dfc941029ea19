"""Host-side checks of the fixed-point element arithmetic (no GPU): C++ programs
compiled with overflow checks compare it with the FP64 elements and a long
double quadrature (tests/host/fx64_check.cpp, fx_vjp_check.cpp, fx_beam_check.cpp)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("check", ["fx64_check", "fx_vjp_check", "fx_beam_check"])
def test_fixed_point_element(check, tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    exe = str(tmp_path / check)
    subprocess.run([gxx, "-std=gnu++17", "-O1", "-fsanitize=signed-integer-overflow", "-fno-sanitize-recover=all",
                    "-Wno-unknown-pragmas", "-I", os.path.join(ROOT, "paper_2103_13890_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host", check + ".cpp"), "-o", exe], check=True,
                   capture_output=True, text=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
    assert out.stdout.startswith("ok")
