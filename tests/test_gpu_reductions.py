"""The reductions' device functions on chosen values: a CUDA program, compiled with
nvcc and linked against libjfnk.so, drives them (tests/host/reduce_check.cu)."""
import os
import subprocess

import pytest

from test_host_tiling import ROOT, _nvcc

pytestmark = pytest.mark.gpu


def test_device_functions(tmp_path):
    from paper_2103_13890_gb300 import build as b
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not found")
    libdir = os.path.dirname(b.LIB)
    exe = str(tmp_path / "reduce_check")
    subprocess.run([nvcc, *b.ARCH, "-std=c++17", "-O1", "--expt-relaxed-constexpr", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2103_13890_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host", "reduce_check.cu"), "-o", exe,
                    "-L", libdir, "-ljfnk", "-Xlinker", "-rpath", "-Xlinker", libdir],
                   check=True, capture_output=True, text=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout + out.stderr
    assert out.stdout.strip() == "ok"
